// k_imex.cu -- cell-local stage of the penalised IMEX Runge-Kutta scheme
// (Sec. 3.4, eq. Bref2 and the scheme after it) and small utility kernels.
//
// Stage l of one cell (one CTA per cell):
//   R_l = f^n + dt sum_{m<l} [ At_lm (G_m/eps - L_m) + A_lm P_m/eps ]
//   U_l = (rho, rho u, E) = discrete moments of R_l                (FP64)
//   M_l = rho (2 pi theta)^(-d/2) exp(-|v - u|^2 / (2 theta))     (parameters FP64)
//   F_l = (R_l + c M_l) / (1 + c),   c = dt A_ll nu / eps
//   P_l = nu (M_l - F_l),   nu = nuf rho (nuf = 1 for BGK, the modes' penalty
//   factor for the Boltzmann model)
// G_l = Q(F_l) - P_l is formed by the inverse-DFT epilogue of the collision
// chain that follows this kernel.
#include <type_traits>

#include "bz_device.cuh"
#include "bz_internal.h"

namespace bz {

namespace {

constexpr int kThreads = 256;

// R_l of one grid point.  The G terms of a step whose G is 0 are left out, and
// in FP64 the terms with a zero coefficient (their buffers need not hold
// anything).  FP32 keeps those: a diverging cell overflows there first, and
// the zero terms carry its NaN to the cells that saw it.
template <typename T>
__device__ __forceinline__ T stage_rhs(const StageCoef &c, T r, const T *__restrict__ G, const T *__restrict__ P,
                                       const T *__restrict__ Lres, int64_t stride, int64_t o, T dt, T ieps) {
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        if (m >= c.nprev) break;
        const int64_t om = (int64_t)m * stride + o;
        if (sizeof(T) == 4 || c.at[m] != 0.0) {
            T gm = c.use_G ? G[om] * ieps : (T)0;
            if (Lres) gm -= Lres[om];
            r = fma(dt * (T)c.at[m], gm, r);
        }
        if (sizeof(T) == 4 || c.a[m] != 0.0) r = fma(dt * (T)c.a[m] * ieps, P[om], r);
    }
    return r;
}

// A number as hi + lo in FP32, and the sum of two such (the high parts' sum exact
// by TwoSum).  round32: such a sum as one FP32 number, the rounded FP64 sum in
// all but rare cases.
__device__ __forceinline__ float2 split32(double x) {
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
}
__device__ __forceinline__ float2 add32(float2 a, float2 b) {
    const float s = a.x + b.x, bb = s - a.x;
    return make_float2(s, ((a.x - (s - bb)) + (b.x - bb)) + (a.y + b.y));
}
__device__ __forceinline__ float round32(float2 a) { return a.x + a.y; }

// Any grid (3-D, and 2-D with N > 32): one CTA per cell.  The Maxwellian is
// formed from one table entry per axis, each axis' N entries formed once per
// cell.  FP64: its factors, pref on the first axis; 2-D, N = 40 on 2000 cells:
// 559 -> 347 us.  FP32: their exponents as (hi, lo), so that a point's exponent is
// the FP64 one rounded once and M takes one exponential (two or three factors
// would round once more each, 0.87e-7 of F's norm for 0.74e-7 at N = 40, 1.03e-7
// for 0.77e-7 in 3-D at N = 16).  A five-stage BGK step on 1406 cells of 40^2 takes
// 953 us (943 with factors, 1428 with FP64 exponents point by point).
template <typename T, int DIM>
__global__ void __launch_bounds__(kThreads) imex_stage_kernel(GridView g, StageCoef c, const T *__restrict__ fn,
                                                              T *__restrict__ F, const T *__restrict__ G,
                                                              T *__restrict__ P, const T *__restrict__ Lres,
                                                              int64_t stride) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *red = reinterpret_cast<double *>(smem_raw);         // 32 * 5
    double *vt = red + 32 * 5;                                   // [N] nodes
    using Entry = typename std::conditional<sizeof(T) == 8, double, float2>::type;
    Entry *fac = reinterpret_cast<Entry *>(vt + g.N);            // [3][N] factors of the Maxwellian, or their exponents
    T *R = reinterpret_cast<T *>(fac + 3 * g.N);                 // nv
    const unsigned N = g.N, nv = (unsigned)g.nv;
    const int64_t base = (int64_t)blockIdx.x * g.nv;
    const T dt = (T)c.dt, ieps = (T)(1.0 / c.eps);
    for (unsigned j = threadIdx.x; j < N; j += blockDim.x) vt[j] = -g.L + (double)j * g.dv;
    __syncthreads();
    double mom[5] = {0, 0, 0, 0, 0};
    for (unsigned i = threadIdx.x; i < nv; i += blockDim.x) {
        const T r = stage_rhs<T>(c, fn[base + i], G, P, Lres, stride, base + i, dt, ieps);
        R[i] = r;
        const double rd = (double)r;
        double v2 = 0.0;
        mom[0] += rd;
        unsigned q = i;
#pragma unroll
        for (int d = DIM - 1; d >= 0; --d) {
            const double vd = vt[q % N];
            q /= N;
            mom[1 + d] = fma(vd, rd, mom[1 + d]);
            v2 = fma(vd, vd, v2);
        }
        mom[DIM + 1] = fma(v2, rd, mom[DIM + 1]);
    }
    block_sum<5>(mom, red);
    double w = 1.0;
    for (int d = 0; d < DIM; ++d) w *= g.dv;
    const double rho = w * mom[0];
    double u[3] = {0, 0, 0}, u2 = 0.0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        u[d] = w * mom[1 + d] / rho;
        u2 += u[d] * u[d];
    }
    const double theta = (w * mom[DIM + 1] / rho - u2) / DIM;
    const double pref = rho * pow(2.0 * M_PI * theta, -0.5 * DIM);
    const double i2t = 0.5 / theta;
    const double nu = c.nuf * rho;
    const double cc = c.dt * c.all * nu / c.eps;
    const T cT = (T)cc, denom = (T)(1.0 / (1.0 + cc)), nuT = (T)nu;
    for (unsigned j = threadIdx.x; j < DIM * N; j += blockDim.x) {
        const int d = (int)(j / N);
        const double o = vt[j % N] - (d == 0 ? u[0] : d == 1 ? u[1] : u[2]);
        if constexpr (sizeof(T) == 8) fac[j] = (d == 0 ? pref : 1.0) * exp(-o * o * i2t);
        else fac[j] = split32(-o * o * i2t);
    }
    __syncthreads();
    T *Fo = F + base;
    T *Po = P + (int64_t)c.stage * stride + base;
    for (unsigned i = threadIdx.x; i < nv; i += blockDim.x) {
        unsigned q = i;
        Entry x = fac[(DIM - 1) * N + q % N];
#pragma unroll
        for (int d = DIM - 2; d >= 0; --d) {
            q /= N;
            if constexpr (sizeof(T) == 8) x *= fac[d * N + q % N];
            else x = add32(x, fac[d * N + q % N]);
        }
        T Mx;
        if constexpr (sizeof(T) == 8) Mx = x;
        else Mx = (T)pref * exp(round32(x));
        const T Fi = (R[i] + cT * Mx) * denom;
        if (c.store_F) Fo[i] = Fi;
        if (c.store_P) Po[i] = nuT * (Mx - Fi);
    }
}

// 2-D, N <= 32: one warp per cell, lane = column j2, loop over rows j1.  (With
// N = 30 in FP64 on 2603 cells the block-per-cell form above took 552 us a
// stage, an exponential and index arithmetic per point on the FP64 pipe.)  FP64
// work is what limits this kernel on a GPU whose FP64 rate is 1/74 of FP32, so
// it is arranged to keep the FP64 pipe's lanes busy with distinct work:
//   * per lane, sums along j1 in the state precision (FP32: with a TwoSum
//     error term), turned into FP64 once (S0, S1, S3 and the v2 products; the
//     error terms stay in FP32);
//   * the 32 lane partials of each cell are summed in FP64 by four threads per
//     (cell, moment) from shared memory, not by a shuffle tree on every lane;
//   * the Maxwellian parameters (rho, u, theta, ...) of the CTA's cells are
//     computed by one warp, one cell per lane, with div64 for the quotients (in
//     FP32 full divisions were the larger part of the kernel's FP64 time);
//   * the Maxwellian of a 2-D grid factorises, M(v1, v2) = pref e1(v1) e2(v2):
//     each lane forms its row and column offsets v - u in FP64 and the rest of
//     the exponent and the exponential in the state precision;
//   * any other N in FP32: dv is no FP32 number, and nodes rounded to FP32 would
//     all lean one way (u_1 off by 3e-7 at N = 30, L = 10).  The sums along j1 are
//     those of R, m R and m^2 R with m = j1 - N/2, whole numbers, each product's
//     error kept by an FMA; dv enters once per cell in FP64.  The exponent of
//     every point is the FP64 one rounded once, as an (hi, lo) sum, and M takes one
//     exponential a point.  A five-stage BGK step, N = 30 on 2500 cells: 151 us
//     (136 with rounded nodes and two factors, 2037 with the block form below and
//     FP64 moments, whose errors these are).
// Mean of a step's stages: FP32 N = 32 on 23160 cells 112 us with full divisions,
// the error terms in FP64 and 8 cells a CTA, 95.5 us now; FP64 N = 30 on 2603
// cells 139 -> 124 us (the row nodes from shared memory, not an FP64 fma per
// row).  Four cells a CTA, so that the warps that wait for the parameters are
// few: 8 cells take 107.6 and 130.5 us.
template <typename T>
__device__ __forceinline__ void acc2(T &s, T &e, T x) {
    if constexpr (sizeof(T) == 4) {
        T t = s + x, bb = t - s;
        e += (s - (t - bb)) + (x - bb);
        s = t;
    } else {
        s += x;
    }
}

constexpr int kStageCells = 4;    // cells (warps) per CTA of the 2-D stage kernel

// NMAX rows in registers; FIXED: N = NMAX at compile time, else any N <= NMAX.
template <typename T, int NMAX, bool FIXED>
__global__ void __launch_bounds__(kStageCells * 32) imex_stage2d_kernel(GridView g, StageCoef c,
                                                                       const T *__restrict__ fn, T *__restrict__ F,
                                                                       const T *__restrict__ G, T *__restrict__ P,
                                                                       const T *__restrict__ Lres, int64_t stride,
                                                                       int64_t n) {
    constexpr bool F32 = sizeof(T) == 4;
    constexpr bool CENTRED = F32 && !FIXED;
    __shared__ double part[kStageCells][4][33];   // per-lane moment partials (pitch 33: no bank conflicts)
    __shared__ T perr[F32 ? kStageCells : 1][F32 ? 4 : 1][33];   // FP32: the partials' error terms
    __shared__ double par[kStageCells][3];        // u1, u2, inv2t
    __shared__ T parT[kStageCells][5];            // nu, inv2t, pref, c, 1/(1+c)
    __shared__ double vd[32];                     // nodes
    __shared__ T vt[F32 ? 1 : 2][F32 ? 1 : NMAX]; // FP64: v1 and v1^2 of the rows
    if (threadIdx.x < 32) {
        vd[threadIdx.x] = -g.L + threadIdx.x * g.dv;
        if (!F32 && threadIdx.x < NMAX) {
            const T v = fma((T)threadIdx.x, (T)g.dv, -(T)g.L);
            vt[0][threadIdx.x] = v;
            vt[!F32][threadIdx.x] = v * v;
        }
    }
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int64_t cell = (int64_t)blockIdx.x * kStageCells + wib;
    const bool live = cell < n;
    const int N = FIXED ? NMAX : g.N, NV = N * N;
    const bool on = lane < N && live;
    const int64_t base = (live ? cell : 0) * NV + (lane < N ? lane : 0);
    const T dt = (T)c.dt, ieps = (T)(1.0 / c.eps);
    T R[NMAX];
#pragma unroll
    for (int j = 0; j < NMAX; ++j) R[j] = on && (FIXED || j < N) ? fn[base + j * N] : (T)0;
#pragma unroll
    for (int m = 0; m < 5; ++m) {              // compile-time index into the coefficient arrays
        if (m >= c.nprev) break;
        const T ca = dt * (T)c.at[m] * ieps, cb = dt * (T)c.a[m] * ieps, cl = dt * (T)c.at[m];
        const int64_t o = (int64_t)m * stride + base;
        // terms left out: as in stage_rhs
        const bool xe = sizeof(T) == 4 || c.at[m] != 0.0;
        const bool ug = xe && c.use_G, up = sizeof(T) == 4 || c.a[m] != 0.0, ul = xe && Lres;
        if (on) {
#pragma unroll
            for (int j = 0; j < NMAX; ++j) {
                if (!FIXED && j >= N) break;
                T r = R[j];
                if (ug) r = fma(ca, G[o + j * N], r);
                if (up) r = fma(cb, P[o + j * N], r);
                if (ul) r = fma(-cl, Lres[o + j * N], r);
                R[j] = r;
            }
        }
    }
    // this lane's partial moments (column j2 = lane)
    __syncthreads();
    {
        T s0 = 0, e0 = 0, s1 = 0, e1 = 0, s3 = 0, e3 = 0;
        const T L = (T)g.L, dv = (T)g.dv;
#pragma unroll
        for (int j = 0; j < NMAX; ++j) {
            T v1, q1;
            if constexpr (!F32) {
                v1 = vt[0][j];
                q1 = vt[1][j];
            } else {
                v1 = CENTRED ? (T)j - (T)(N / 2) : fma((T)j, dv, -L);
                q1 = v1 * v1;
            }
            acc2(s0, e0, R[j]);
            const T x1 = v1 * R[j], x3 = q1 * R[j];
            if constexpr (CENTRED) {
                e1 += fma(v1, R[j], -x1);
                e3 += fma(q1, R[j], -x3);
            }
            acc2(s1, e1, x1);
            acc2(s3, e3, x3);
        }
        const double vv = vd[lane], S0 = (double)s0;
        part[wib][0][lane] = S0;
        part[wib][1][lane] = (double)s1;
        part[wib][2][lane] = vv * S0;
        part[wib][3][lane] = fma(vv * vv, S0, CENTRED ? g.dv * g.dv * (double)s3 : (double)s3);
        if constexpr (F32) {                 // of relative size 2^-24: their sums in FP32 lose nothing
            const T v = (T)vv;
            perr[wib][0][lane] = e0;
            perr[wib][1][lane] = e1;
            perr[wib][2][lane] = v * e0;
            perr[wib][3][lane] = fma(v * v, e0, CENTRED ? dv * dv * e3 : e3);
        }
    }
    __syncthreads();
    // sums over the 32 lanes of each cell: four threads per (cell, moment) sum
    // eight partials each, then combine by shuffles (a fixed order)
    if (threadIdx.x < kStageCells * 16) {
        const int cc = threadIdx.x >> 4, q = (threadIdx.x >> 2) & 3, pp = threadIdx.x & 3;
        double tot = 0.0;
#pragma unroll
        for (int l = 0; l < 8; ++l) tot += part[cc][q][pp * 8 + l];
        if constexpr (F32) {
            T te = (T)0;
#pragma unroll
            for (int l = 0; l < 8; ++l) te += perr[cc][q][pp * 8 + l];
            tot += (double)te;
        }
        tot += __shfl_xor_sync(0xffffffffu, tot, 1);
        tot += __shfl_xor_sync(0xffffffffu, tot, 2);
        if (pp == 0) part[cc][q][32] = tot;
    }
    __syncthreads();
    // Maxwellian parameters, one cell per lane of warp 0
    if (threadIdx.x < kStageCells) {
        const int cc = threadIdx.x;
        const double w = g.dv * g.dv, coef = c.coef;
        const double S0 = part[cc][0][32];
        double S1 = part[cc][1][32], S3 = part[cc][3][32];
        if constexpr (CENTRED) {             // v = c0 + m dv
            const double c0 = fma((double)(N / 2), g.dv, -g.L), m1 = g.dv * S1;
            S1 = fma(c0, S0, m1);
            S3 = fma(c0, fma(c0, S0, 2.0 * m1), S3);
        }
        const double rho = w * S0, yr = rcp64(rho);
        const double u1 = div64(w * S1, rho, yr), u2 = div64(w * part[cc][2][32], rho, yr);
        const double E = 0.5 * w * S3;
        const double theta = (div64(2.0 * E, rho, yr) - (u1 * u1 + u2 * u2)) * 0.5, yt = rcp64(theta);
        const double cst = coef * rho, c1 = 1.0 + cst;
        par[cc][0] = u1;
        par[cc][1] = u2;
        par[cc][2] = div64(0.5, theta, yt);
        parT[cc][0] = (T)(c.nuf * rho);    // penalty rate nu
        parT[cc][1] = (T)par[cc][2];
        parT[cc][2] = (T)div64(rho * (0.5 / M_PI), theta, yt);
        parT[cc][3] = (T)cst;
        parT[cc][4] = (T)div64(1.0, c1, rcp64(c1));
    }
    __syncthreads();
    if (!live) return;
    // separable Maxwellian: this lane's column factor and row factor j1 = lane;
    // offsets v - u in FP64, the rest of the exponent and the exp in T
    // (any other N: the whole exponent in FP64; FP32: one exponential a point)
    const double vl = vd[lane];
    const double d2 = vl - par[wib][1], d1 = vl - par[wib][0];
    T fcol = (T)0, frow_l = (T)0;
    float2 xcol = make_float2(0.f, 0.f), xrow = xcol;
    if constexpr (FIXED) {
        const T i2t = parT[wib][1], t1 = (T)d1, t2 = (T)d2;
        fcol = parT[wib][2] * exp(-t2 * t2 * i2t);
        frow_l = exp(-t1 * t1 * i2t);
    } else if constexpr (F32) {
        xcol = split32(-d2 * d2 * par[wib][2]);
        xrow = split32(-d1 * d1 * par[wib][2]);
    } else {
        fcol = parT[wib][2] * exp(-d2 * d2 * par[wib][2]);
        frow_l = exp(-d1 * d1 * par[wib][2]);
    }
    const T cT = parT[wib][3], denom = parT[wib][4], nuT = parT[wib][0];
    T *Fo = F + base;
    T *Po = P + (int64_t)c.stage * stride + base;
#pragma unroll
    for (int j = 0; j < NMAX; ++j) {
        if (!FIXED && j >= N) break;
        T Mx;
        if constexpr (CENTRED) {
            const float2 xr = make_float2(__shfl_sync(0xffffffffu, xrow.x, j), __shfl_sync(0xffffffffu, xrow.y, j));
            Mx = parT[wib][2] * exp(round32(add32(xcol, xr)));
        } else {
            Mx = fcol * __shfl_sync(0xffffffffu, frow_l, j);
        }
        const T Fi = (R[j] + cT * Mx) * denom;
        if (on) {
            if (c.store_F) Fo[j * N] = Fi;
            if (c.store_P) Po[j * N] = nuT * (Mx - Fi);
        }
    }
}

template <typename T>
__global__ void check_input_kernel(const T *__restrict__ f, int64_t count, int *err) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t step = (int64_t)gridDim.x * blockDim.x;
    bool bad = false;
    for (; i < count; i += step) bad |= !isfinite(f[i]);
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) raise_device_error(err, kDevNonFinite);
}

template <typename T>
cudaError_t stage(const GridView &g, const StageCoef &c, const T *fn, T *F, const T *G, T *P,
                  const T *Lres, int64_t stride, int64_t n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (g.dim == 2 && g.N <= 32) {
        const unsigned blocks = (unsigned)((n + kStageCells - 1) / kStageCells);
        const unsigned thr = kStageCells * 32;
        if (g.N == 16) imex_stage2d_kernel<T, 16, true><<<blocks, thr, 0, st>>>(g, c, fn, F, G, P, Lres, stride, n);
        else if (g.N == 24) imex_stage2d_kernel<T, 24, true><<<blocks, thr, 0, st>>>(g, c, fn, F, G, P, Lres, stride, n);
        else if (g.N == 32) imex_stage2d_kernel<T, 32, true><<<blocks, thr, 0, st>>>(g, c, fn, F, G, P, Lres, stride, n);
        else imex_stage2d_kernel<T, 32, false><<<blocks, thr, 0, st>>>(g, c, fn, F, G, P, Lres, stride, n);
        return cudaGetLastError();
    }
    const size_t sm = sizeof(double) * (32 * 5 + 4 * g.N) + sizeof(T) * (size_t)g.nv;
    auto *kern = g.dim == 2 ? imex_stage_kernel<T, 2> : imex_stage_kernel<T, 3>;
    cudaError_t e = allow_dynamic_smem((const void *)kern, sm);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)n, kThreads, sm, st>>>(g, c, fn, F, G, P, Lres, stride);
    return cudaGetLastError();
}

template <typename T> cudaError_t check(const T *f, int64_t count, int *err, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    int64_t blocks = (count + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    check_input_kernel<T><<<(unsigned)blocks, 256, 0, st>>>(f, count, err);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_imex_stage_f64(const GridView &g, const StageCoef &c, const double *fn, double *F,
                                  const double *G, double *P, const double *Lres, int64_t stride,
                                  int64_t n, cudaStream_t st) {
    return stage<double>(g, c, fn, F, G, P, Lres, stride, n, st);
}
cudaError_t launch_imex_stage_f32(const GridView &g, const StageCoef &c, const float *fn, float *F,
                                  const float *G, float *P, const float *Lres, int64_t stride,
                                  int64_t n, cudaStream_t st) {
    return stage<float>(g, c, fn, F, G, P, Lres, stride, n, st);
}
cudaError_t launch_check_input_f64(const double *f, int64_t count, int *err, cudaStream_t st) {
    return check<double>(f, count, err, st);
}
cudaError_t launch_check_input_f32(const float *f, int64_t count, int *err, cudaStream_t st) {
    return check<float>(f, count, err, st);
}
cudaError_t launch_fill_zero(void *p, int64_t bytes, cudaStream_t st) {
    if (bytes <= 0) return cudaSuccess;
    return cudaMemsetAsync(p, 0, (size_t)bytes, st);
}

}  // namespace bz
