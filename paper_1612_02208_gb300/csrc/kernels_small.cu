// Levels 1 and 0 of the V-cycle (Alg. 1 below the second-coarsest grid) in ONE thread block.
//
// With the paper's coarsest grid (8 x 8) level 1 is 16 x 16: 768 unknowns.  Run as separate
// kernels, its smoothing sweeps, IB passes, residual, restriction, the dense coarsest solve and the
// prolongation are a chain of 11 (Vanka) to 45 (Schur complement) dependent launches, each costing
// a launch and a round trip to L2 for almost no work.  Here one block of 1024 threads keeps the
// whole level in shared memory -- iterates, right-hand side, IB force, the patch entries, the SC
// diagonals and the assembled IB windows -- and separates the same steps by __syncthreads().
// The set-up data is copied in before the wait on the preceding kernel; only the right-hand side
// is read after it, and only the level's solution is written back.
//
// Every step evaluates the same point-wise formulas as the per-level kernels (grid_cells.cuh),
// in the same order, on shared-memory copies of the same arrays.
#include <cooperative_groups.h>

#include <algorithm>

#include "grid_cells.cuh"

namespace cg = cooperative_groups;

namespace sib {

namespace {

template <typename T>
struct SmallSmem {
    T *x, *xt, *b, *r, *fib, *pf, *dinv, *pd;
    T *y, *d, *gq, *ya, *gq2, *dA2, *dA, *sv, *dp, *dM;
    T *b0, *x0, *win;
    int* tiles;
    unsigned char* tile;
};

// shared-memory layout of block 0: T arrays (the Vanka patch corrections share their space with
// the SC temporaries), then the active-tile list, then the tile flags
template <typename T>
__host__ __device__ inline size_t small_layout(int n, int n0, int nTiles, int per, int ntiles, SmallSmem<T>* s,
                                               unsigned char* base) {
    size_t off = 0;
    SmallSmem<T> dummy;
    SmallSmem<T>* q = s ? s : &dummy;
    auto take = [&](T** p, size_t cnt) {
        *p = reinterpret_cast<T*>(base + off);
        off += sizeof(T) * cnt;
    };
    take(&q->x, 3 * n);
    take(&q->xt, 3 * n);
    take(&q->b, 3 * n);
    take(&q->r, 3 * n);
    take(&q->fib, 2 * n);
    take(&q->pf, 7 * n);
    take(&q->dinv, 3 * n);
    const size_t tmp = off;   // SC temporaries, or the Vanka corrections (5 n <= 17 n)
    take(&q->y, 2 * n);
    take(&q->d, 2 * n);
    take(&q->gq, 2 * n);
    take(&q->ya, 2 * n);
    take(&q->gq2, 2 * n);
    take(&q->dA2, 2 * n);
    take(&q->dA, 2 * n);
    take(&q->sv, n);
    take(&q->dp, n);
    take(&q->dM, n);
    q->pd = reinterpret_cast<T*>(base + tmp);
    take(&q->b0, n0);
    take(&q->x0, n0);
    take(&q->win, (size_t)nTiles * 2 * WIN_SIZE * per);
    off = (off + 15) & ~(size_t)15;
    q->tiles = reinterpret_cast<int*>(base + off);
    off += sizeof(int) * (size_t)(nTiles > 0 ? nTiles : 1);
    q->tile = base + off;
    off += (size_t)ntiles;
    return (off + 15) & ~(size_t)15;
}

constexpr int NT = 1024;

__device__ __forceinline__ int ilog2(int v) { return 31 - __clz(v); }
constexpr int SMALL_CLUSTER = 8;

// Block-wide copy of `bytes` (a multiple of 16; both addresses 16-byte aligned) in 16-byte words,
// eight loads in flight per thread before their stores.
__device__ __forceinline__ void block_copy16(void* dst, const void* src, size_t bytes) {
    constexpr int U = 8;
    const int4* __restrict__ s = static_cast<const int4*>(src);
    int4* __restrict__ d = static_cast<int4*>(dst);
    const size_t n = bytes / 16;
    for (size_t q0 = 0; q0 < n; q0 += (size_t)NT * U) {
        int4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t q = q0 + threadIdx.x + (size_t)u * NT;
            if (q < n) v[u] = s[q];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t q = q0 + threadIdx.x + (size_t)u * NT;
            if (q < n) d[q] = v[u];
        }
    }
}


// f = [S K J] u on the active tiles: one thread per (slot, component, face), window rows summed in
// the per-level kernel's order.  Tile sizes, tile counts and N are powers of two: index arithmetic
// by shifts.  (The pass is bound by shared-memory bandwidth: 81 coefficients and 81 values a face.)
template <typename T>
__device__ void sm_ib(const GridK<T>& g, const SmallSmem<T>& s, int nTiles, const T* u, T* f) {
    const int N = g.N, lgN = ilog2(N), mk = N - 1, lgtx = g.lgtx, lgty = g.lgty;
    const int lgper = lgtx + lgty, per = 1 << lgper, lgntx = lgN - lgtx;
    const int items = nTiles * 2 * per;
    for (int item = threadIdx.x; item < items; item += NT) {
        const int q = item & (per - 1), rest = item >> lgper;
        const int c = rest & 1, slot = rest >> 1;
        const int t = s.tiles[slot];
        const int i = ((t & ((1 << lgntx) - 1)) << lgtx) + (q & ((1 << lgtx) - 1));
        const int j = ((t >> lgntx) << lgty) + (q >> lgtx);
        const T* w = s.win + (((slot * 2 + c) * WIN_SIZE) << lgper) + q;
        const T* uc = u + (c << (2 * lgN));
        T sum = T(0);
#pragma unroll
        for (int r = 0; r < WD; ++r) {
            const T* row = uc + (((j + r - WR) & mk) << lgN);
            T acc = T(0);
#pragma unroll
            for (int ox = -WR; ox <= WR; ++ox) acc += w[(r * WD + ox + WR) << lgper] * row[(i + ox) & mk];
            sum += acc;
        }
        f[(c << (2 * lgN)) + (j << lgN) + i] = sum;
    }
}

// one additive Vanka sweep xo = x + omega sum_c W_c R_c^T L_c^{-1} R_c (b - L x) (x == nullptr:
// zero start); g.fib holds [SKJ] x
template <typename T>
__device__ void sm_vanka(const GridK<T>& g, const SmallSmem<T>& s, const T* x, const T* b, T* xo) {
    const int N = g.N, n = N * N, m = N - 1;
    for (int c = threadIdx.x; c < n; c += NT) {
        const int i = c & m, j = c >> ilog2(N);
        if (x) {
            s.r[c] = res_u(g, x, b, i, j);
            s.r[n + c] = res_v(g, x, b, i, j);
            s.r[2 * n + c] = res_p(g, x, b, i, j);
        } else {
            s.r[c] = b[c];
            s.r[n + c] = b[n + c];
            s.r[2 * n + c] = b[2 * n + c];
        }
    }
    __syncthreads();
    const T ih = g.inv_h;
    for (int c = threadIdx.x; c < n; c += NT) {
        const int i = c & m, j = c >> ilog2(N);
        const int ce = j * N + ((i + 1) & m), cn = ((j + 1) & m) * N + i;
        const T r0 = s.r[c], r1 = s.r[ce], r2 = s.r[n + c], r3 = s.r[n + cn], r4 = s.r[2 * n + c];
        T f[7];
#pragma unroll
        for (int k = 0; k < 7; ++k) f[k] = g.pf[k * n + c];   // the cell's set-up patch factors
        T d0, d1, d2, d3, dp;
        patch_solve(f, ih, r0, r1, r2, r3, r4, d0, d1, d2, d3, dp);
        s.pd[c] = d0;
        s.pd[n + c] = d1;
        s.pd[2 * n + c] = d2;
        s.pd[3 * n + c] = d3;
        s.pd[4 * n + c] = dp;
    }
    __syncthreads();
    const T hw = T(0.5) * g.omega;
    for (int c = threadIdx.x; c < n; c += NT) {
        const int i = c & m, j = c >> ilog2(N);
        const int cw = j * N + ((i - 1) & m), cs = ((j - 1) & m) * N + i;
        const T du = hw * (s.pd[c] + s.pd[n + cw]);
        const T dv = hw * (s.pd[2 * n + c] + s.pd[3 * n + cs]);
        const T dq = g.omega * s.pd[4 * n + c];
        xo[c] = x ? x[c] + du : du;
        xo[n + c] = x ? x[n + c] + dv : dv;
        xo[2 * n + c] = x ? x[2 * n + c] + dq : dq;
    }
    __syncthreads();
}

// one Schur-complement sweep with two Chebyshev iterations per inner solve (x == nullptr: zero start)
template <typename T>
__device__ void sm_sc(const GridK<T>& g, const SmallArgs<T>& a, const SmallSmem<T>& s, const T* x, const T* b,
                      T* xo) {
    const int N = g.N, n = N * N, m = N - 1;
    const bool ib = a.nTiles > 0 && g.tile != nullptr;
    T* fib = const_cast<T*>(g.fib);
    if (x && ib) {
        sm_ib(g, s, a.nTiles, x, fib);
        __syncthreads();
    }
    for (int c = threadIdx.x; c < n; c += NT) sc_start_cell(g, a.ka, x, b, s.r, s.d, c & m, c >> ilog2(N), sc_pre<T, false>(g, c & m, c >> ilog2(N)));
    __syncthreads();
    if (ib) {
        sm_ib(g, s, a.nTiles, s.d, fib);
        __syncthreads();
    }
    for (int c = threadIdx.x; c < n; c += NT) sc_chebA_cell(g, a.ka, s.r, s.d, s.y, c & m, c >> ilog2(N), sc_pre<T, false>(g, c & m, c >> ilog2(N)));
    __syncthreads();
    for (int c = threadIdx.x; c < n; c += NT)
        sc_mstart_cell(g, a.ka, a.km, s.r + 2 * n, s.y, s.sv, s.dM, s.gq, s.dA, c & m, c >> ilog2(N),
                       sc_pre<T, true>(g, c & m, c >> ilog2(N)));
    __syncthreads();
    if (ib) {
        sm_ib(g, s, a.nTiles, s.dA, fib);
        __syncthreads();
    }
    for (int c = threadIdx.x; c < n; c += NT) sc_chebA_cell(g, a.ka, s.gq, s.dA, s.ya, c & m, c >> ilog2(N), sc_pre<T, false>(g, c & m, c >> ilog2(N)));
    __syncthreads();
    for (int c = threadIdx.x; c < n; c += NT)
        sc_mfinish_cell(g, a.ka, a.km, s.sv, s.dM, s.ya, s.dp, s.gq2, s.dA2, c & m, c >> ilog2(N),
                        sc_pre<T, true>(g, c & m, c >> ilog2(N)));
    __syncthreads();
    if (ib) {
        sm_ib(g, s, a.nTiles, s.dA2, fib);
        __syncthreads();
    }
    for (int c = threadIdx.x; c < n; c += NT) sc_finish_cell(g, a.ka, x, s.y, s.gq2, s.dA2, s.dp, xo, c & m, c >> ilog2(N),
                       sc_pre<T, false>(g, c & m, c >> ilog2(N)));
    __syncthreads();
}

template <typename T>
__device__ void sm_sweep(const GridK<T>& g, const SmallArgs<T>& a, const SmallSmem<T>& s, const T* x, const T* b,
                         T* xo) {
    if (a.smoother == SIB_SMOOTHER_SC) {
        sm_sc(g, a, s, x, b, xo);
        return;
    }
    if (x && a.nTiles > 0 && g.tile != nullptr) {
        sm_ib(g, s, a.nTiles, x, const_cast<T*>(g.fib));
        __syncthreads();
    }
    sm_vanka(g, s, x, b, xo);
}

// Block 0 runs level 1; blocks 1 .. csize-1 hold slices of the coarsest pseudo-inverse in shared
// memory (loaded before the wait) and apply it when block 0 has formed b0: each reads b0 from
// block 0's shared memory and writes its rows of x0 there, between two cluster barriers.
template <typename T>
__device__ void coarse_helper(const SmallArgs<T>& a, unsigned char* smraw, cg::cluster_group& cl) {
    const int rank = (int)cl.block_rank(), nh = (int)cl.num_blocks() - 1;
    const int rows = (a.n0 + nh - 1) / nh;
    const int r0 = (rank - 1) * rows, r1 = r0 + rows < a.n0 ? r0 + rows : a.n0;
    double* P = reinterpret_cast<double*>(smraw);                 // rows r0 .. r1-1
    double* bl = P + (size_t)rows * a.n0;                         // local copy of b0
    if (r1 > r0) block_copy16(P, a.Pinv + (size_t)r0 * a.n0, sizeof(double) * (size_t)(r1 - r0) * a.n0);
    pdl_entry();
    __syncthreads();
    SmallSmem<T> lay;
    const int N = a.g.N;
    small_layout<T>(N * N, a.n0, a.nTiles, a.g.tx * a.g.ty, a.ntiles, &lay, smraw);
    cl.sync();   // b0 formed by block 0
    const T* b0 = cl.map_shared_rank(lay.b0, 0);
    T* x0 = cl.map_shared_rank(lay.x0, 0);
    for (int c = threadIdx.x; c < a.n0; c += NT) bl[c] = (double)b0[c];
    __syncthreads();
    // four lanes a row: strided partial sums, then two butterfly steps.  The loop runs over
    // groups of eight rows, one group per warp, so every lane of a warp takes the same trip count
    // and reaches the shuffles; lanes of rows past r1 contribute nothing and store nothing.
    const int sub = threadIdx.x & 3;
    for (int rb = r0 + (int)(threadIdx.x >> 5) * 8; rb < r1; rb += (NT / 32) * 8) {
        const int r = rb + (int)((threadIdx.x & 31) >> 2);
        double acc = 0.0;
        if (r < r1) {
            const double* row = P + (size_t)(r - r0) * a.n0;
            for (int c = sub; c < a.n0; c += 4) acc += row[c] * bl[c];
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if (sub == 0 && r < r1) x0[r] = (T)acc;
    }
    cl.sync();   // x0 complete in block 0
}

template <typename T>
__global__ void __launch_bounds__(NT, 1) k_vcycle_small(const __grid_constant__ SmallArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    cg::cluster_group cl = cg::this_cluster();
    if (cl.block_rank() != 0) {
        coarse_helper(a, smraw, cl);
        return;
    }
    const GridK<T>& G = a.g;
    const int N = G.N, n = N * N, per = G.tx * G.ty;
    SmallSmem<T> s;
    small_layout<T>(n, a.n0, a.nTiles, per, a.ntiles, &s, smraw);
    // set-up data: not written by the kernels this one waits for (every array is a multiple of
    // 16 bytes: n is a multiple of 16)
    if (a.smoother == SIB_SMOOTHER_VANKA) block_copy16(s.pf, G.pf, sizeof(T) * 7 * n);
    if (a.smoother == SIB_SMOOTHER_SC) block_copy16(s.dinv, G.dinv, sizeof(T) * 3 * n);
    if (a.nTiles > 0) block_copy16(s.win, a.win, sizeof(T) * (size_t)a.nTiles * 2 * WIN_SIZE * per);
    for (int q = threadIdx.x; q < a.nTiles; q += NT) s.tiles[q] = a.tiles[q];
    if (G.tile)
        for (int q = threadIdx.x; q < a.ntiles; q += NT) s.tile[q] = G.tile[q];
    pdl_entry();
    block_copy16(s.b, a.b, sizeof(T) * 3 * n);
    __syncthreads();
    GridK<T> g = G;
    g.fib = s.fib;
    g.pf = s.pf;
    g.dinv = s.dinv;
    g.tile = G.tile ? s.tile : nullptr;
    const bool ib = a.nTiles > 0 && g.tile != nullptr;
    const int m = N - 1;

    T* x = s.x;
    T* xt = s.xt;
    int k0 = 0;
    if (a.nu1 > 0) {
        sm_sweep(g, a, s, (const T*)nullptr, s.b, xt);   // first sweep from w = 0
        T* t = x;
        x = xt;
        xt = t;
        k0 = 1;
    } else {
        for (int q = threadIdx.x; q < 3 * n; q += NT) x[q] = T(0);
        __syncthreads();
    }
    for (int k = k0; k < a.nu1; ++k) {
        sm_sweep(g, a, s, x, s.b, xt);
        T* t = x;
        x = xt;
        xt = t;
    }
    if (ib) {
        sm_ib(g, s, a.nTiles, x, s.fib);
        __syncthreads();
    }
    const int Nc = N / 2;
    for (int c = threadIdx.x; c < n; c += NT) {
        const int i = c & m, j = c >> ilog2(N);
        s.r[c] = res_u(g, x, s.b, i, j);
        s.r[n + c] = res_v(g, x, s.b, i, j);
        s.r[2 * n + c] = res_p(g, x, s.b, i, j);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < Nc * Nc; c += NT) restrict_cell(Nc, (const T*)s.r, s.b0, c & (Nc - 1), c >> ilog2(Nc));
    __syncthreads();
    cl.sync();   // b0 to the helpers
    cl.sync();   // x0 = Pinv b0 back from them
    for (int c = threadIdx.x; c < n; c += NT) prolong_add_cell(Nc, (const T*)s.x0, x, c & m, c >> ilog2(N));
    __syncthreads();
    for (int k = 0; k < a.nu2; ++k) {
        sm_sweep(g, a, s, x, s.b, xt);
        T* t = x;
        x = xt;
        xt = t;
    }
    block_copy16(a.out, x, sizeof(T) * 3 * n);
}

// ------------------------------------------------------------------------------------------
// The levels of up to 32 x 32 cells and the coarsest solve in one cluster of eight blocks (FP32, Vanka).
//
// As separate launches a 32 x 32 level is ten dependent kernels of 2 to 3 us, and k_vcycle_small runs 16 x 16
// on one SM while seven wait: together 53 of the 133 us of a 128^2 solve's iteration.  Here every level is cut into
// eight strips of rows, one per block, held in shared memory with the strip's patch factors and IB windows; a
// neighbour's row is read from its block's shared memory, and a step ends with a cluster barrier (two a
// sweep).  Bound by the latency of those steps and barriers, about 0.3 us each; eight blocks are the portable
// cluster, and with them a block's share of a full 32 x 32 level's windows, 83 KB, fits beside the rest.
// 32^2 ellipse: solve 1.51 -> 1.16 ms; 128^2 disk: 2.53 -> 2.33 ms (the windows still copied through registers; cp.async since).
// The formulas are those of the per-level kernels in the same order.  FP64 levels keep the kernels above: eight
// SMs' FP64 pipes are slower than the launches.
constexpr int CV_T = 576, CV_WR8 = 2 * WR;   // 576: nine window rows of the 64 face vectors of a 32 x 32 strip
__device__ __forceinline__ const float* cv_at(cg::cluster_group& cl, float* p, int rank) {
    return cl.map_shared_rank(p, rank);
}

// 16 bytes to shared memory without a stop in a register (zero without `real`)
__device__ __forceinline__ void cv_copy16(void* dst, const void* src, bool real) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(real ? 16 : 0)
                 : "memory");
}

// r = b - L x on the block's strip
__device__ __forceinline__ void cv_residual(cg::cluster_group& cl, const ClusterArgs& a, const ClusterLevel& L, float* sm,
                                            int rank) {
    const int N = L.N, m = N - 1, R = N / SMALL_CLUSTER, RN = R * N, lgR = L.lgN - 3, j0 = rank * R;
    const float* part = sm + a.part;
    if (L.ib) {   // u and v with a halo of WR, then the window rows of four faces a thread
        const int W = N + CV_WR8, H = R + CV_WR8, nf = 2 * RN;
        float* uh = sm + a.uh;
        for (int t = threadIdx.x; t < 2 * H * W; t += CV_T) {
            const int c = t >= H * W, q = t - c * H * W, jj = q / W, j = (j0 - WR + jj) & m, i = (q - jj * W - WR) & m;
            uh[t] = *cv_at(cl, sm + L.x + c * RN + ((j & (R - 1)) << L.lgN) + i, j >> lgR);
        }
        __syncthreads();
        for (int t = threadIdx.x; t < WD * nf / 4; t += CV_T) {
            const int oy = t / (nf / 4), f = (t - oy * (nf / 4)) * 4, c = f >= RN, q = f - c * RN;
            const int lj = q >> L.lgN, i = q & m;
            const float4* u4 = reinterpret_cast<const float4*>(uh + (c * H + lj + oy) * W + i);
            float u[4 + CV_WR8];
#pragma unroll
            for (int v = 0; v < (4 + CV_WR8) / 4; ++v) {
                const float4 x = u4[v];
                u[4 * v] = x.x, u[4 * v + 1] = x.y, u[4 * v + 2] = x.z, u[4 * v + 3] = x.w;
            }
            const float* w = sm + L.wins + (size_t)oy * WD * nf + f;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int ox = 0; ox < WD; ++ox) {
                const float4 k = *reinterpret_cast<const float4*>(w + ox * nf);
                acc.x += k.x * u[ox], acc.y += k.y * u[ox + 1], acc.z += k.z * u[ox + 2], acc.w += k.w * u[ox + 3];
            }
            *reinterpret_cast<float4*>(sm + a.part + oy * nf + f) = acc;
        }
        __syncthreads();
    }
    const float* xl = sm + L.x;
    const float* bl = sm + L.b;
    for (int t = threadIdx.x; t < RN; t += CV_T) {
        const int lj = t >> L.lgN, i = t & m, e = lj * N + ((i + 1) & m), w = lj * N + ((i - 1) & m);
        const float* xn = lj + 1 < R ? xl + t + N : cv_at(cl, sm + L.x + i, (rank + 1) & (SMALL_CLUSTER - 1));
        const float* xs = lj > 0 ? xl + t - N : cv_at(cl, sm + L.x + (R - 1) * N + i, (rank - 1) & (SMALL_CLUSTER - 1));
        const float u = xl[t], v = xl[RN + t], p = xl[2 * RN + t], uE = xl[e], vN = xn[RN];
        float Au = L.a0 * u - L.c * ((uE + xl[w]) + (xn[0] + xs[0])) + (p - xl[2 * RN + w]) * L.ih;
        float Av = L.a0 * v - L.c * ((xl[RN + e] + xl[RN + w]) + (vN + xs[RN])) + (p - xs[2 * RN]) * L.ih;
        if (L.ib) {
            float fu = 0.f, fv = 0.f;
#pragma unroll
            for (int k = 0; k < WD; ++k) fu += part[k * 2 * RN + t], fv += part[k * 2 * RN + RN + t];
            Au -= L.dt * fu;
            Av -= L.dt * fv;
        }
        float* r = sm + L.r + t;
        r[0] = bl[t] - Au;
        r[RN] = bl[RN + t] - Av;
        r[2 * RN] = bl[2 * RN + t] + ((uE - u) + (vN - v)) * L.ih;
    }
}

// x += omega times the weighted patch corrections of the residual at rr (x = them: zero).  A cell takes the patches
// of its own, its western and its southern cell.
__device__ __forceinline__ void cv_update(cg::cluster_group& cl, const ClusterArgs& a, const ClusterLevel& L, float* sm,
                                          int rank, int rr, bool zero) {
    const int N = L.N, m = N - 1, R = N / SMALL_CLUSTER, RN = R * N;
    const float* rl = sm + rr;
    const float hw = 0.5f * a.omega;
    for (int t = threadIdx.x; t < RN; t += CV_T) {
        const int lj = t >> L.lgN, i = t & m, ie = (i + 1) & m, iw = (i - 1) & m;
        const float* rc = rl + lj * N;
        const float* rn = lj + 1 < R ? rc + N : cv_at(cl, sm + rr, (rank + 1) & (SMALL_CLUSTER - 1));
        const float* rs = lj > 0 ? rc - N : cv_at(cl, sm + rr + (R - 1) * N, (rank - 1) & (SMALL_CLUSTER - 1));
        float f[3][7];
        const float* pf = sm + L.pfs + lj * N;   // row lj of the strip's factors is the row to the south
#pragma unroll
        for (int k = 0; k < 7; ++k) {
            const float* pk = pf + k * (RN + N);
            f[0][k] = pk[N + i], f[1][k] = pk[N + iw], f[2][k] = pk[i];
        }
        const float ru = rc[i], rv = rc[RN + i];
        float d0, d1, d2, d3, dp, w0, w1, w2, w3, wp, s0, s1, s2, s3, sp;
        patch_solve(f[0], L.ih, ru, rc[ie], rv, rn[RN + i], rc[2 * RN + i], d0, d1, d2, d3, dp);
        patch_solve(f[1], L.ih, rc[iw], ru, rc[RN + iw], rn[RN + iw], rc[2 * RN + iw], w0, w1, w2, w3, wp);
        patch_solve(f[2], L.ih, rs[i], rs[ie], rs[RN + i], rv, rs[2 * RN + i], s0, s1, s2, s3, sp);
        const float du = hw * (d0 + w1), dv = hw * (d2 + s3), dq = a.omega * dp;
        float* x = sm + L.x + t;
        x[0] = zero ? du : x[0] + du;
        x[RN] = zero ? dv : x[RN] + dv;
        x[2 * RN] = zero ? dq : x[2 * RN] + dq;
    }
}

// sum of the six (u, v) or four (p) residual terms that coarse cell (I, J) restricts; row(c, j) gives row j of component c
template <typename Row>
__device__ __forceinline__ float cv_restrict(int comp, int I, int J, int m, Row row) {
    const int i = 2 * I, j = 2 * J, ip = i + 1, im = (i - 1) & m;
    const float *q = row(comp, j), *qn = row(comp, j + 1);
    if (comp == 0) return 0.25f * ((q[i] + qn[i]) + 0.5f * ((q[ip] + qn[ip]) + (q[im] + qn[im])));
    if (comp == 2) return 0.25f * ((q[i] + q[ip]) + (qn[i] + qn[ip]));
    const float* qs = row(comp, (j - 1) & m);
    return 0.25f * ((q[i] + q[ip]) + 0.5f * ((qn[i] + qn[ip]) + (qs[i] + qs[ip])));
}

__global__ void __launch_bounds__(CV_T, 1) k_vcycle_cluster(const __grid_constant__ ClusterArgs a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    cg::cluster_group cl = cg::this_cluster();
    float* sm = reinterpret_cast<float*>(smraw);
    const int rank = (int)cl.block_rank(), top = a.levels - 1;
    // set-up data: not written by the kernel this one waits for
    for (int l = 0; l <= top; ++l) {
        const ClusterLevel& L = a.lv[l];
        const int N = L.N, m = N - 1, R = N / SMALL_CLUSTER, RN = R * N, j0 = rank * R;
        for (int t = threadIdx.x * 4; t < 7 * (RN + N); t += CV_T * 4) {
            const int k = t / (RN + N), q = t - k * (RN + N);
            cv_copy16(sm + L.pfs + t, L.pf + k * N * N + (((j0 - 1 + (q >> L.lgN)) & m) << L.lgN) + (q & m), true);
        }
        if (!L.ib) continue;
        const int nv = 2 * RN / 4;   // 16-byte vectors of four faces (at most 64); CV_T / nv threads share one's entries
        const int f = (threadIdx.x & (nv - 1)) * 4, c = f >= RN, q = f - c * RN, j = j0 + (q >> L.lgN), i = q & m;
        const int slot = L.slotOf[((j >> L.lgty) << L.lgntx) + (i >> L.lgtx)];
        const float* w = L.win + (((size_t)((slot < 0 ? 0 : slot) * 2 + c) * WIN_SIZE) << (L.lgtx + L.lgty)) +
                         ((j & ((1 << L.lgty) - 1)) << L.lgtx) + (i & ((1 << L.lgtx) - 1));
        for (int k = threadIdx.x / nv; k < WIN_SIZE; k += CV_T / nv)
            cv_copy16(sm + L.wins + k * 2 * RN + f, w + ((size_t)k << (L.lgtx + L.lgty)), slot >= 0);
    }
    const int prows = a.n0 / SMALL_CLUSTER;   // rows of the pseudo-inverse per block
    double* P = reinterpret_cast<double*>(sm + a.P);
    for (int t = threadIdx.x * 2; t < prows * a.n0; t += CV_T * 2)
        cv_copy16(P + t, a.Pinv + (size_t)rank * prows * a.n0 + t, true);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    pdl_entry();
    {
        const ClusterLevel& L = a.lv[top];
        const int RN = L.N / SMALL_CLUSTER * L.N, n = L.N * L.N;
        for (int t = threadIdx.x; t < 3 * RN; t += CV_T) {
            const int c = t / RN;
            sm[L.b + t] = a.b[c * n + rank * RN + t - c * RN];
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    cl.sync();
    auto sweep = [&](const ClusterLevel& L) {
        cv_residual(cl, a, L, sm, rank);
        cl.sync();
        cv_update(cl, a, L, sm, rank, L.r, false);
    };
    for (int l = top; l >= 0; --l) {
        const ClusterLevel& L = a.lv[l];
        const int N = L.N, R = N / SMALL_CLUSTER, RN = R * N, lgR = L.lgN - 3, m = N - 1, Nc = N / 2;
        if (a.nu1 > 0) {
            cv_update(cl, a, L, sm, rank, L.b, true);   // from zero the residual is b
        } else {
            for (int t = threadIdx.x; t < 3 * RN; t += CV_T) sm[L.x + t] = 0.f;
        }
        cl.sync();
        for (int k = 1; k < a.nu1; ++k) {
            sweep(L);
            cl.sync();
        }
        cv_residual(cl, a, L, sm, rank);
        cl.sync();
        auto row = [&](int c, int j) { return cv_at(cl, sm + L.r + c * RN + ((j & (R - 1)) << L.lgN), j >> lgR); };
        if (l > 0) {
            const ClusterLevel& C = a.lv[l - 1];
            const int Rc = R / 2, RNc = Rc * Nc;
            for (int t = threadIdx.x; t < 3 * RNc; t += CV_T) {
                const int c = t / RNc, q = t - c * RNc, lJ = q >> C.lgN;
                sm[C.b + t] = cv_restrict(c, q & (Nc - 1), rank * Rc + lJ, m, row);
            }
            cl.sync();
            continue;
        }
        // coarsest solve: the whole b0 in every block, a share of the rows each, the result to all
        double* b0 = reinterpret_cast<double*>(sm + a.b0);
        const int nc = Nc * Nc;
        for (int t = threadIdx.x; t < a.n0; t += CV_T) {
            const int c = t / nc, q = t - c * nc;
            b0[t] = (double)cv_restrict(c, q & (Nc - 1), q / Nc, m, row);
        }
        __syncthreads();
        const int sub = threadIdx.x & 7;   // eight lanes a row; every lane of a warp takes the same trips
        for (int r0 = 0; r0 < prows; r0 += CV_T / 8) {
            const int r = r0 + (int)(threadIdx.x >> 3);
            double acc = 0.0;
            if (r < prows)
                for (int c = sub; c < a.n0; c += 8) acc += P[r * a.n0 + c] * b0[c];
            for (int o = 1; o < 8; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (r < prows) *cl.map_shared_rank(sm + a.x0 + rank * prows + r, sub) = (float)acc;
        }
        cl.sync();
    }
    for (int l = 0; l <= top; ++l) {
        const ClusterLevel& L = a.lv[l];
        const ClusterLevel& C = a.lv[l > 0 ? l - 1 : 0];
        const int N = L.N, m = N - 1, R = N / SMALL_CLUSTER, RN = R * N, Nc = N / 2, mc = Nc - 1;
        const int Rc = l > 0 ? R / 2 : Nc, lgNc = L.lgN - 1, lgRc = l > 0 ? L.lgN - 4 : lgNc, RNc = Rc * Nc;
        for (int t = threadIdx.x; t < RN; t += CV_T) {
            const int i = t & m, j = rank * R + (t >> L.lgN), I = i >> 1, J = j >> 1;
            const int I1 = (I + 1) & mc, I2 = (I + ((i & 1) ? 1 : -1)) & mc, J2 = (J + ((j & 1) ? 1 : -1)) & mc;
            // coarse rows J and J2: x0 is whole in every block, a coarser level's strip in its own
            const float* e = l > 0 ? cv_at(cl, sm + C.x + ((J & (Rc - 1)) << lgNc), J >> lgRc) : sm + a.x0 + J * Nc;
            const float* e2 = l > 0 ? cv_at(cl, sm + C.x + ((J2 & (Rc - 1)) << lgNc), J2 >> lgRc) : sm + a.x0 + J2 * Nc;
            const float pu = (i & 1) ? 0.5f * (e[I] + e[I1]) : e[I];
            const float pv = (j & 1) ? 0.5f * (e[RNc + I] + e2[RNc + I]) : e[RNc + I];
            const float pp = 9.0f / 16.0f * e[2 * RNc + I] + 3.0f / 16.0f * (e[2 * RNc + I2] + e2[2 * RNc + I]) +
                             1.0f / 16.0f * e2[2 * RNc + I2];
            float* x = sm + L.x + t;
            x[0] += pu;
            x[RN] += pv;
            x[2 * RN] += pp;
        }
        for (int k = 0; k < a.nu2; ++k) {
            cl.sync();
            sweep(L);
        }
        if (l == top) {   // every thread writes the cells that it updated last
            const int n = N * N;
            for (int t = threadIdx.x; t < RN; t += CV_T)
                for (int c = 0; c < 3; ++c) a.out[c * n + rank * RN + t] = sm[L.x + c * RN + t];
        }
        cl.sync();   // for the finer level's prolongation; no block leaves while another reads its shared memory
    }
}

}  // namespace

size_t cluster_layout(ClusterArgs& a) {
    int off = 0, halo = 0, part = 0;
    auto take = [&](int n) {
        const int p = off;
        off += (n + 3) & ~3;
        return p;
    };
    for (int l = 0; l < a.levels; ++l) {
        ClusterLevel& L = a.lv[l];
        const int R = L.N / SMALL_CLUSTER, RN = R * L.N;
        L.x = take(3 * RN);
        L.b = take(3 * RN);
        L.r = take(3 * RN);
        L.pfs = take(7 * (RN + L.N));
        L.wins = take(L.ib ? WIN_SIZE * 2 * RN : 0);
        if (!L.ib) continue;
        halo = std::max(halo, 2 * (R + CV_WR8) * (L.N + CV_WR8));
        part = std::max(part, WD * 2 * RN);
    }
    a.uh = take(halo);
    a.part = take(part);
    a.x0 = take(a.n0);
    a.b0 = take(2 * a.n0);
    a.P = take(2 * (a.n0 / SMALL_CLUSTER) * a.n0);
    return sizeof(float) * (size_t)off;
}
static cudaLaunchConfig_t cluster_config(size_t smem, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(SMALL_CLUSTER);
    cfg.blockDim = dim3(CV_T);
    cfg.dynamicSmemBytes = smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = SMALL_CLUSTER;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}
bool vcycle_cluster_fits(size_t smem) {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cluster_config(smem, attr);
    cfg.numAttrs = 1;
    int clusters = 0;
    if (allow_smem(k_vcycle_cluster, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, k_vcycle_cluster, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return clusters > 0;
}
cudaError_t launch_vcycle_cluster(const ClusterArgs& a, size_t smem, cudaStream_t s) {
    cudaError_t e = allow_smem(k_vcycle_cluster, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cluster_config(smem, attr);
    cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, k_vcycle_cluster, a);
}

template <typename T>
size_t vcycle_small_smem(int N1, int n0, int nTiles, int per, int ntiles) {
    return small_layout<T>(N1 * N1, n0, nTiles, per, ntiles, nullptr, nullptr);
}

// Cluster size of the launch: block 0 and the coarse-solve helpers (8, the portable maximum), 0
// if such a cluster cannot be resident with `smem` bytes per block.
template <typename T>
int vcycle_small_cluster(size_t smem) {
    if (allow_smem(k_vcycle_small<T>, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(SMALL_CLUSTER);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = SMALL_CLUSTER;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, k_vcycle_small<T>, &cfg) != cudaSuccess || clusters < 1) {
        cudaGetLastError();
        return 0;
    }
    return SMALL_CLUSTER;
}

template <typename T>
cudaError_t launch_vcycle_small(const SmallArgs<T>& a, size_t smem, cudaStream_t s) {
    cudaError_t e = allow_smem(k_vcycle_small<T>, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(SMALL_CLUSTER);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = SMALL_CLUSTER;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k_vcycle_small<T>, a);
}

template size_t vcycle_small_smem<float>(int, int, int, int, int);
template size_t vcycle_small_smem<double>(int, int, int, int, int);
template int vcycle_small_cluster<float>(size_t);
template int vcycle_small_cluster<double>(size_t);
template cudaError_t launch_vcycle_small<float>(const SmallArgs<float>&, size_t, cudaStream_t);
template cudaError_t launch_vcycle_small<double>(const SmallArgs<double>&, size_t, cudaStream_t);

}  // namespace sib
