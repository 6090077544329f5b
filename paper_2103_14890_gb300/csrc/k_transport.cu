// k_transport.cu -- transport residual of the finite-volume scheme (Sec. 3.2,
// eq. finite_vol5 / eq. ho): CWENO reconstruction of degree 1 or 2 and Rusanov
// fluxes, for every cell and every discrete velocity of a 2-D grid.
//
// Layout: f, L are [cell][nv] (the collision operator's layout), so one
// cell's velocities are contiguous.  A block takes up to 1024 velocities of
// one cell: every table entry of the cell is a warp-uniform load and every f
// access a coalesced row segment (neighbour rows come from L2: a 32^2 grid of
// 20k cells holds 81 MB in FP32).  Cells are taken along a Morton curve of
// their barycentres; every table is stored in that order.
//
// Orders 2 and 3 take two passes.  For a linear flux v f the Rusanov flux
//   F = (v.n)(f_L + f_R)/2 - |v.n| (f_R - f_L)/2
// is the upwind flux (v.n) f_L for v.n > 0 and (v.n) f_R for v.n < 0, and v.n
// is constant along a straight face, so the face integral needs one mean of
// the reconstruction per face (midpoint for degree 1, two Gauss points for
// degree 2), on the upwind side only.
//   Pass 1 reconstructs the polynomial of every (cell, velocity) in registers
//   and writes its mean over a face, for the velocities that leave the cell
//   there, into that face's row, FX [face][nv]; the cell on the other side of
//   the face writes the others.  Both sides form v.n from the same normal up to
//   its sign (table fs), so every entry is written exactly once (v.n = 0: by
//   the owner).  Boundary faces are transmissive: their cell writes every
//   velocity.
//   Pass 2 sums v.n times a cell's face rows by FMA, the normals its own (table
//   fn), and divides by |P_i|.
// FP64 rows hold the flux (v.n times the mean) instead, and pass 2 adds them up:
// the product and the normal velocity would take as long again (0.106 ms for
// 0.050 on 2603 cells x 30^2) and gain no accuracy.  The exception are faces whose
// two copies, a period apart in a periodic mesh, differ by rounding (kFvSplit):
// with one side's normal for both, a cell's normals no longer sum to zero (errors
// on 300 and 1200 Voronoi cells 2.2e-15 and 3.3e-15 of L's norm, 1.1e-15 and
// 1.2e-15 with its own).
// FP32, thin cells (kFvThin; slivers of a Delaunay triangulation along the
// boundary, half a percent of the cells): the fluxes cancel to L by a factor
// of hundreds to thousands, which turns a rounding into a visible change of L.
// Pass 1 also writes both sides' values at their faces (rows after the flux
// rows, one per Gauss point), and pass 2 sums the two-sided Rusanov form there,
// so that such cells keep the rounding they had with it (and, should they
// overflow in an unstable run, their neighbours see it on every velocity).
// Against gradients or coefficients in memory and both sides' states at every
// face this halves the traffic on triangles (1.5 rows written and read per
// cell in place of 5 and 24 for degree 2) and cuts the arithmetic that bounds
// FP64 (the GB300 does 2 FP64 operations per clock and SM): per hexagon face
// and velocity 9 operations in place of 34.  19802 triangles x 32^2, FP32,
// degree 2: 0.382 -> 0.238 ms; 2603 Voronoi cells x 30^2, FP64, degree 2: 2.13
// -> 1.34 ms, 1.20 with p_0's rows and one difference per neighbour in the
// cells flagged kFvRegular (pass 1 1.27 -> 1.13 ms, the FP64 pipe nine tenths
// busy), 1.03 with signs, comparisons and 1 / #sectors off that pipe (pass 1
// 0.98 ms, sums 0.070 -> 0.050).
//
// Reconstruction: the central (least-squares) coefficients and the sector
// polynomials are linear in the averages (tables Rc, Rs of fv_mesh.cpp);
// p_0 = (p_opt - lambda_L sum_L p_L) / lambda_0 (lambda_0 = 3/4, lambda_L =
// 1/4 / #sectors); smoothness sigma_s = h^2 |grad p_s|^2 (degree 2: the cell
// mean, plus the squared scaled second derivatives); weights
// proportional to lambda_s / (sigma_s + eps)^4 with eps = 1e-14, formed as
// lambda_s ((sigma_min + eps) / (sigma_s + eps))^4 so that no power
// underflows in FP32.
//
// Order 1 (piecewise constant) needs no reconstruction: one pass.
#include <algorithm>
#include <atomic>

#include "bz_device.cuh"
#include "bz_internal.h"

namespace bz {

namespace {

constexpr int kFvThreads = 256;

// VEC consecutive velocities per thread, all in one row of the velocity grid
// (N is even, and the host takes VEC = 4 only when 4 divides N): the cell's
// table entries are loaded once for all of them and f moves in 8- or 16-byte
// vectors (the host checks the alignment, else VEC = 1).
template <typename T, int VEC> struct Vec {
    T v[VEC];
};
template <typename T, int VEC>
__device__ __forceinline__ Vec<T, VEC> ldv(const T *__restrict__ p) {
    Vec<T, VEC> r;
    if constexpr (VEC == 2) {
        const typename C2<T>::type q = *reinterpret_cast<const typename C2<T>::type *>(p);
        r.v[0] = q.x; r.v[1] = q.y;
    } else if constexpr (VEC == 4 && sizeof(T) == 4) {
        const float4 q = *reinterpret_cast<const float4 *>(p);
        r.v[0] = q.x; r.v[1] = q.y; r.v[2] = q.z; r.v[3] = q.w;
    } else if constexpr (VEC == 4 && sizeof(T) == 8) {
        const double2 q0 = reinterpret_cast<const double2 *>(p)[0], q1 = reinterpret_cast<const double2 *>(p)[1];
        r.v[0] = q0.x; r.v[1] = q0.y; r.v[2] = q1.x; r.v[3] = q1.y;
    } else {
#pragma unroll
        for (int u = 0; u < VEC; ++u) r.v[u] = p[u];
    }
    return r;
}
// The same for what the kernel before wrote, in a kernel launched after it
// programmatically (see griddep_wait).
template <typename T, int VEC>
__device__ __forceinline__ Vec<T, VEC> ldv_after(const T *p) {
    Vec<T, VEC> r;
    if constexpr (VEC == 2) {
        const typename C2<T>::type q = __ldcg(reinterpret_cast<const typename C2<T>::type *>(p));
        r.v[0] = q.x; r.v[1] = q.y;
    } else if constexpr (VEC == 4 && sizeof(T) == 4) {
        const float4 q = __ldcg(reinterpret_cast<const float4 *>(p));
        r.v[0] = q.x; r.v[1] = q.y; r.v[2] = q.z; r.v[3] = q.w;
    } else {
#pragma unroll
        for (int u = 0; u < VEC; ++u) r.v[u] = __ldcg(p + u);
    }
    return r;
}
template <typename T, int VEC>
__device__ __forceinline__ void stv(T *__restrict__ p, const Vec<T, VEC> &r) {
    if constexpr (VEC == 2) {
        *reinterpret_cast<typename C2<T>::type *>(p) = cmk<typename C2<T>::type>(r.v[0], r.v[1]);
    } else if constexpr (VEC == 4 && sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4(r.v[0], r.v[1], r.v[2], r.v[3]);
    } else if constexpr (VEC == 4 && sizeof(T) == 8) {
        reinterpret_cast<double2 *>(p)[0] = make_double2(r.v[0], r.v[1]);
        reinterpret_cast<double2 *>(p)[1] = make_double2(r.v[2], r.v[3]);
    } else {
#pragma unroll
        for (int u = 0; u < VEC; ++u) p[u] = r.v[u];
    }
}

// four values off any 16-byte boundary
template <typename T> __device__ __forceinline__ Vec<T, 4> ld4(const T *__restrict__ p) {
    Vec<T, 4> r;
#pragma unroll
    for (int u = 0; u < 4; ++u) r.v[u] = p[u];
    return r;
}

// FP32x2 arithmetic on pairs of velocities: one FADD2 / FMUL2 / FFMA2 rounds
// each lane as its scalar instruction does.
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 lo2(const float4 &a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ float2 hi2(const float4 &a) { return make_float2(a.z, a.w); }
// approximate reciprocal (1 ulp; the argument is a normal number here)
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(rcp_approx(a.x), rcp_approx(a.y)); }

// Index tables of a mesh by position p of the processing order (bz_mesh).
struct FvIdx {
    const int *order, *meta, *fid, *two, *ncen, *cen, *nsec, *sec;
};

// Signs and comparisons of finite FP64 values as integers, off the FP64 pipe.
__device__ __forceinline__ bool positive(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool positive(float x) { return x > 0.f; }
__device__ __forceinline__ double negate_if(bool neg, double x) {
    return __hiloint2double(__double2hiint(x) ^ (neg ? 0x80000000 : 0), __double2loint(x));
}
// Not negative (-0 included), for a velocity, never a NaN.
template <typename T> __device__ __forceinline__ bool leaves(T vn) {
    if constexpr (sizeof(T) == 8) return !positive(negate_if(true, vn));
    else return vn >= (T)0;
}

// Write a face's row where this cell is upwind (everywhere on a boundary face):
// the reconstructed mean `val` of VEC velocities, vn their outward normal
// velocities; flux (FP64): vn times it, in the owner's orientation.
template <typename T, int VEC>
__device__ __forceinline__ void put_upwind(T *__restrict__ row, const T (&vn)[VEC], const T (&val)[VEC], bool other,
                                           bool boundary, bool flux) {
    Vec<T, VEC> o;
    bool on[VEC], all = true;
#pragma unroll
    for (int u = 0; u < VEC; ++u) {
        o.v[u] = val[u];
        if constexpr (sizeof(T) == 8)
            if (flux) o.v[u] = negate_if(other, vn[u] * val[u]);
        on[u] = boundary || (other ? positive(vn[u]) : leaves(vn[u]));
        all = all && on[u];
    }
    if (all) {
        stv<T, VEC>(row, o);
    } else {
#pragma unroll
        for (int u = 0; u < VEC; ++u)
            if (on[u]) row[u] = o.v[u];
    }
}

// Normal velocities v . |e|n of VEC velocities of one grid row (explicit FMA:
// every path rounds alike, so the two sides of a face agree up to the sign).
template <typename T, int VEC>
__device__ __forceinline__ void normal_velocity(T v1, const T (&v2)[VEC], T nx, T ny, T (&vn)[VEC]) {
    const T a = v1 * nx;
    if constexpr (sizeof(T) == 4 && VEC == 4) {
#pragma unroll
        for (int h = 0; h < 4; h += 2) {
            const float2 x = fma2(make_float2(v2[h], v2[h + 1]), dup2(ny), dup2(a));
            vn[h] = x.x;
            vn[h + 1] = x.y;
        }
    } else {
#pragma unroll
        for (int u = 0; u < VEC; ++u) vn[u] = fma(v2[u], ny, a);
    }
}

// lambda_L = 1/4 / #sectors (a division costs as much as ten FMAs)
static_assert(kFvMaxFaces == 8, "entries of kLamSector");
__constant__ double kLamSector[kFvMaxFaces + 1] = {0.0,      0.25,     0.25 / 2, 0.25 / 3, 0.25 / 4,
                                                   0.25 / 5, 0.25 / 6, 0.25 / 7, 0.25 / 8};

// Coefficients of a cell's CWENO polynomial in FP64, one velocity per thread
// (any polygon).  B, K: coefficients and stencil cells (2, 5 or 5, 11); MAXS
// bounds the sectors.  Loops are unrolled with block-uniform predicates.
template <int MAXS, int B, int K>
__device__ __forceinline__ void recon_coefs_f64(const double *__restrict__ f, const FvTables<double> &tb,
                                                const FvIdx &ix, int64_t p, int ncf, int k, int nv, double fi,
                                                double (&c)[B]) {
#pragma unroll
    for (int l = 0; l < B; ++l) c[l] = 0.0;
    const int nc = ncf & (kFvRegular - 1), ns = __ldg(ix.nsec + p);
    const double *Rc = tb.Rc + p * (B * K), *Rs = tb.Rs + p * kFvMaxFaces * 4;
    constexpr double kLam0 = 0.75, kEps = 1e-14;
    const double lamL = kLamSector[ns];
    double sx[MAXS], sy[MAXS];
    if (ncf & kFvRegular) {              // uniform over the block; the rows of p_0, the sectors' share included
        double d[MAXS];
#pragma unroll
        for (int q = 0; q < K; ++q) {
            const double dq = f[(int64_t)__ldg(ix.cen + p * K + q) * nv + k] - fi;
            if (q < MAXS) d[q] = dq;
#pragma unroll
            for (int l = 0; l < B; ++l) c[l] = fma(__ldg(Rc + l * K + q), dq, c[l]);
        }
#pragma unroll
        for (int s = 0; s < MAXS; ++s)
            if (s < ns) {
                const double db = s + 1 < ns ? d[(s + 1) % MAXS] : d[0];
                sx[s] = fma(__ldg(Rs + 4 * s), d[s], __ldg(Rs + 4 * s + 1) * db);
                sy[s] = fma(__ldg(Rs + 4 * s + 2), d[s], __ldg(Rs + 4 * s + 3) * db);
            }
    } else {
#pragma unroll
        for (int q = 0; q < K; ++q) {
            if (q < nc) {
                const double d = f[(int64_t)__ldg(ix.cen + p * K + q) * nv + k] - fi;
#pragma unroll
                for (int l = 0; l < B; ++l) c[l] = fma(__ldg(Rc + l * K + q), d, c[l]);
            }
        }
        if (ns == 0) return;
        double sumx = 0.0, sumy = 0.0;
#pragma unroll
        for (int s = 0; s < MAXS; ++s) {
            if (s < ns) {
                const int a = __ldg(ix.sec + (p * kFvMaxFaces + s) * 2), b = __ldg(ix.sec + (p * kFvMaxFaces + s) * 2 + 1);
                const double da = f[(int64_t)a * nv + k] - fi, db = f[(int64_t)b * nv + k] - fi;
                sx[s] = fma(__ldg(Rs + 4 * s), da, __ldg(Rs + 4 * s + 1) * db);
                sy[s] = fma(__ldg(Rs + 4 * s + 2), da, __ldg(Rs + 4 * s + 3) * db);
                sumx += sx[s];
                sumy += sy[s];
            }
        }
        // p_0's coefficients (1 / lambda_0 is in Rc)
        const double lam10 = lamL * (4.0 / 3.0);
        c[0] = fma(-lam10, sumx, c[0]);
        c[1] = fma(-lam10, sumy, c[1]);
    }
    // sigma + eps of every polynomial
    double s0 = fma(c[0], c[0], fma(c[1], c[1], kEps));
    if constexpr (B == kFvCoef3) {
        const double *q = tb.quad + 4 * p;
        const double q3 = __ldg(q + 3);
        s0 = fma(c[2], fma(__ldg(q), c[2], q3 * c[3]), s0);
        s0 = fma(c[3], fma(__ldg(q + 1), c[3], q3 * c[4]), s0);
        s0 = fma(c[4], __ldg(q + 2) * c[4], s0);
    }
    double sig[MAXS];
    int least = __double2hiint(s0);
#pragma unroll
    for (int s = 0; s < MAXS; ++s)
        if (s < ns) {
            sig[s] = fma(sx[s], sx[s], fma(sy[s], sy[s], kEps));
            least = min(least, __double2hiint(sig[s]));
        }
    // weights (2^e / (sigma + eps))^4, 2^e the power of two below the least of them
    const int scale = (least & 0x7ff00000) - 0x3ff00000;
    double r = scaled_rcp(s0, scale);
    r = r * r;
    double w = kLam0 * (r * r), wl = 0.0, ax = 0.0, ay = 0.0;
#pragma unroll
    for (int s = 0; s < MAXS; ++s)
        if (s < ns) {
            r = scaled_rcp(sig[s], scale);
            r = r * r;
            r = r * r;
            wl += r;
            ax = fma(r, sx[s], ax);
            ay = fma(r, sy[s], ay);
        }
    // (lambda_0 w_0 p_0 + lambda_L sum w_L p_L) / (lambda_0 w_0 + lambda_L sum w_L)
    const double iw = rcp64(fma(lamL, wl, w)), wL = lamL * iw;
    w *= iw;
#pragma unroll
    for (int l = 0; l < B; ++l) c[l] *= w;
    c[0] = fma(wL, ax, c[0]);
    c[1] = fma(wL, ay, c[1]);
}

// The same coefficients in FP32.
template <int VEC, int MAXS>
__device__ __forceinline__ void recon_coefs_f32(const float *__restrict__ f, const FvTables<float> &tb, const FvIdx &ix,
                                                int64_t p, int ncf, int k, int nv, const Vec<float, VEC> &fi,
                                                float (&c)[2][VEC]) {
    const int nc = ncf & (kFvRegular - 1), ns = __ldg(ix.nsec + p);
    // central least-squares gradient
    float gx[VEC], gy[VEC];
    {
        Vec<float, VEC> fj[kFvCentral];
        float rx[kFvCentral], ry[kFvCentral];
#pragma unroll
        for (int q = 0; q < kFvCentral; ++q) {
            rx[q] = ry[q] = (float)0;
            fj[q] = fi;
            if (q < nc) {
                const int j = __ldg(ix.cen + p * kFvCentral + q);
                rx[q] = __ldg(tb.Rc + (p * 2) * kFvCentral + q);
                ry[q] = __ldg(tb.Rc + (p * 2 + 1) * kFvCentral + q);
                fj[q] = ldv<float, VEC>(f + (int64_t)j * nv + k);
            }
        }
#pragma unroll
        for (int u = 0; u < VEC; ++u) {
            gx[u] = gy[u] = (float)0;
#pragma unroll
            for (int q = 0; q < kFvCentral; ++q) {
                const float d = fj[q].v[u] - fi.v[u];
                gx[u] += rx[q] * d;
                gy[u] += ry[q] * d;
            }
        }
    }
    if (ns > 0) {
        constexpr float kLam0 = (float)0.75, kInvLam0 = (float)(4.0 / 3.0), kEps = (float)1e-14;
        const float lamL = (float)0.25 / (float)ns, h2 = __ldg(tb.quad + 4 * p + 3);
        float sx[MAXS][VEC], sy[MAXS][VEC];
        {
            Vec<float, VEC> fa[MAXS], fb[MAXS];
            float R[MAXS][4];
#pragma unroll
            for (int s = 0; s < MAXS; ++s) {
                fa[s] = fi;
                fb[s] = fi;
                R[s][0] = R[s][1] = R[s][2] = R[s][3] = (float)0;
                if (s < ns) {
                    const int a = __ldg(ix.sec + (p * kFvMaxFaces + s) * 2), b = __ldg(ix.sec + (p * kFvMaxFaces + s) * 2 + 1);
                    const float *Rp = tb.Rs + (p * kFvMaxFaces + s) * 4;
#pragma unroll
                    for (int c = 0; c < 4; ++c) R[s][c] = __ldg(Rp + c);
                    fa[s] = ldv<float, VEC>(f + (int64_t)a * nv + k);
                    fb[s] = ldv<float, VEC>(f + (int64_t)b * nv + k);
                }
            }
#pragma unroll
            for (int s = 0; s < MAXS; ++s)
#pragma unroll
                for (int u = 0; u < VEC; ++u) {
                    const float da = fa[s].v[u] - fi.v[u], db = fb[s].v[u] - fi.v[u];
                    sx[s][u] = R[s][0] * da + R[s][1] * db;
                    sy[s][u] = R[s][2] * da + R[s][3] * db;
                }
        }
#pragma unroll
        for (int u = 0; u < VEC; ++u) {
            float sumx = (float)0, sumy = (float)0;
#pragma unroll
            for (int s = 0; s < MAXS; ++s)
                if (s < ns) {
                    sumx += sx[s][u];
                    sumy += sy[s][u];
                }
            const float g0x = (gx[u] - lamL * sumx) * kInvLam0, g0y = (gy[u] - lamL * sumy) * kInvLam0;
            const float sig0 = h2 * (g0x * g0x + g0y * g0y);
            float sig[MAXS];
            float smin = sig0;
#pragma unroll
            for (int s = 0; s < MAXS; ++s) {
                sig[s] = h2 * (sx[s][u] * sx[s][u] + sy[s][u] * sy[s][u]);
                if (s < ns) smin = fmin(smin, sig[s]);
            }
            // fast divisions (2 ulp; the weights are smooth in sigma)
            const float num = smin + kEps;
            float r = __fdividef(num, sig0 + kEps);
            r = r * r;
            float w = kLam0 * (r * r);
            float wsum = w, ax = w * g0x, ay = w * g0y;
#pragma unroll
            for (int s = 0; s < MAXS; ++s)
                if (s < ns) {
                    r = __fdividef(num, sig[s] + kEps);
                    r = r * r;
                    w = lamL * (r * r);
                    wsum += w;
                    ax += w * sx[s][u];
                    ay += w * sy[s][u];
                }
            const float iw = (float)1 / wsum;
            gx[u] = ax * iw;
            gy[u] = ay * iw;
        }
    }
#pragma unroll
    for (int u = 0; u < VEC; ++u) {
        c[0][u] = gx[u];
        c[1][u] = gy[u];
    }
}
template <int VEC, int MAXS>
__device__ __forceinline__ void recon_coefs_f32(const float *__restrict__ f, const FvTables<float> &tb, const FvIdx &ix,
                                                int64_t p, int ncf, int k, int nv, const Vec<float, VEC> &fi,
                                                float (&c)[kFvCoef3][VEC]) {
#pragma unroll
    for (int l = 0; l < kFvCoef3; ++l)
#pragma unroll
        for (int u = 0; u < VEC; ++u) c[l][u] = 0.f;
    const int nc = ncf & (kFvRegular - 1);
    const float *Rc = tb.Rc + p * kFvCoef3 * kFvCentral3;
#pragma unroll
    for (int q = 0; q < kFvCentral3; ++q) {
        if (q < nc) {
            const int j = __ldg(ix.cen + p * kFvCentral3 + q);
            const Vec<float, VEC> fj = ldv<float, VEC>(f + (int64_t)j * nv + k);
#pragma unroll
            for (int l = 0; l < kFvCoef3; ++l) {
                const float r = __ldg(Rc + l * kFvCentral3 + q);
#pragma unroll
                for (int u = 0; u < VEC; ++u) c[l][u] += r * (fj.v[u] - fi.v[u]);
            }
        }
    }
    const int ns = __ldg(ix.nsec + p);
    if (ns > 0) {
        constexpr float kInvLam0 = (float)(4.0 / 3.0), kLam0 = (float)0.75, kEps = (float)1e-14;
        const float lamL = (float)0.25 / (float)ns;
        float sx[MAXS][VEC], sy[MAXS][VEC];
#pragma unroll
        for (int s = 0; s < MAXS; ++s) {
#pragma unroll
            for (int u = 0; u < VEC; ++u) sx[s][u] = sy[s][u] = (float)0;
            if (s < ns) {
                const int a = __ldg(ix.sec + (p * kFvMaxFaces + s) * 2), b = __ldg(ix.sec + (p * kFvMaxFaces + s) * 2 + 1);
                const float *R = tb.Rs + (p * kFvMaxFaces + s) * 4;
                const float r0 = __ldg(R), r1 = __ldg(R + 1), r2 = __ldg(R + 2), r3 = __ldg(R + 3);
                const Vec<float, VEC> fa = ldv<float, VEC>(f + (int64_t)a * nv + k), fb = ldv<float, VEC>(f + (int64_t)b * nv + k);
#pragma unroll
                for (int u = 0; u < VEC; ++u) {
                    const float da = fa.v[u] - fi.v[u], db = fb.v[u] - fi.v[u];
                    sx[s][u] = r0 * da + r1 * db;
                    sy[s][u] = r2 * da + r3 * db;
                }
            }
        }
        const float m20 = __ldg(tb.quad + 4 * p), m11 = __ldg(tb.quad + 4 * p + 1), m02 = __ldg(tb.quad + 4 * p + 2);
#pragma unroll
        for (int u = 0; u < VEC; ++u) {
            float sumx = (float)0, sumy = (float)0;
#pragma unroll
            for (int s = 0; s < MAXS; ++s) {
                sumx += sx[s][u];
                sumy += sy[s][u];
            }
            float p0[kFvCoef3];
            p0[0] = (c[0][u] - lamL * sumx) * kInvLam0;
            p0[1] = (c[1][u] - lamL * sumy) * kInvLam0;
#pragma unroll
            for (int l = 2; l < kFvCoef3; ++l) p0[l] = c[l][u] * kInvLam0;
            const float sig0 = p0[0] * p0[0] + p0[1] * p0[1] + (float)4 * p0[2] * p0[2] * m20 + (float)4 * p0[2] * p0[3] * m11 +
                           p0[3] * p0[3] * m02 + p0[3] * p0[3] * m20 + (float)4 * p0[3] * p0[4] * m11 +
                           (float)4 * p0[4] * p0[4] * m02 + (float)4 * p0[2] * p0[2] + p0[3] * p0[3] + (float)4 * p0[4] * p0[4];
            float sig[MAXS], smin = sig0;
#pragma unroll
            for (int s = 0; s < MAXS; ++s) {
                sig[s] = sx[s][u] * sx[s][u] + sy[s][u] * sy[s][u];
                if (s < ns) smin = fmin(smin, sig[s]);
            }
            const float num = smin + kEps;
            float r = __fdividef(num, sig0 + kEps);
            r = r * r;
            float w = kLam0 * (r * r);
            float wsum = w, acc[kFvCoef3];
#pragma unroll
            for (int l = 0; l < kFvCoef3; ++l) acc[l] = w * p0[l];
#pragma unroll
            for (int s = 0; s < MAXS; ++s)
                if (s < ns) {
                    r = __fdividef(num, sig[s] + kEps);
                    r = r * r;
                    w = lamL * (r * r);
                    wsum += w;
                    acc[0] += w * sx[s][u];
                    acc[1] += w * sy[s][u];
                }
            const float iw = (float)1 / wsum;
#pragma unroll
            for (int l = 0; l < kFvCoef3; ++l) c[l][u] = acc[l] * iw;
        }
    }
}

// A table value: in global memory, or staged in shared memory (SM).
template <bool SM, typename X> __device__ __forceinline__ X tab_load(const X *p) {
    if constexpr (SM) return *p;
    else return __ldg(p);
}

// f + sum_l c_l phi_l for VEC velocities.
template <typename T, int VEC, int B, bool SM = false>
__device__ __forceinline__ void point_value(const Vec<T, VEC> &fi, const T (&c)[B][VEC], const T *__restrict__ phi,
                                            T (&val)[VEC]) {
    if constexpr (sizeof(T) == 4 && VEC == 4) {
        float2 x = make_float2(fi.v[0], fi.v[1]), y = make_float2(fi.v[2], fi.v[3]);
#pragma unroll
        for (int l = 0; l < B; ++l) {
            const float2 ph = dup2(tab_load<SM>(phi + l));
            x = fma2(make_float2(c[l][0], c[l][1]), ph, x);
            y = fma2(make_float2(c[l][2], c[l][3]), ph, y);
        }
        val[0] = x.x; val[1] = x.y; val[2] = y.x; val[3] = y.y;
    } else {
#pragma unroll
        for (int u = 0; u < VEC; ++u) val[u] = fi.v[u];
#pragma unroll
        for (int l = 0; l < B; ++l) {
            const T ph = tab_load<SM>(phi + l);
#pragma unroll
            for (int u = 0; u < VEC; ++u) val[u] = fma(c[l][u], ph, val[u]);
        }
    }
}

// Rows of a two-sided face behind the flux rows: [face][side][Gauss point].
template <int B> __device__ __forceinline__ int64_t two_row(int64_t rows, int two, int side, int g) {
    constexpr int GP = B == kFvCoef3 ? 2 : 1;
    return rows + ((int64_t)two * 2 + side) * GP + g;
}

// Face q of the cell at position p: its mean for the velocities it is upwind of,
// and on a two-sided face (FP32) the values at its points.  fs, phi: the face's
// entries of these tables.
// TWO: only the values at its two points (every face taken as two-sided; the
// rows number faces).
template <typename T, int VEC, int B, bool SM, bool TWO = false>
__device__ __forceinline__ void emit_face(T *__restrict__ FX, const FvTables<T> &tb, const FvIdx &ix, int64_t rows,
                                          int64_t p, int q, int fid, int meta, int k, int nv, T v1,
                                          const T (&v2)[VEC], const Vec<T, VEC> &fi, const T (&c)[B][VEC],
                                          const T *fs, const T *phi) {
    const int64_t s = p * kFvMaxFaces + q;
    T vn[VEC], val[VEC];
    const bool other = (meta >> (8 + q)) & 1, boundary = (meta >> (16 + q)) & 1;
    if (TWO || (sizeof(T) == 4 && ((meta >> (24 + q)) & 1))) {
        const int two = TWO ? fid : __ldg(ix.two + s) & (kFvSplit - 1);
#pragma unroll
        for (int g = 0; g < (B == kFvCoef3 ? 2 : 1); ++g) {
            point_value<T, VEC, B>(fi, c, B == kFvCoef3 ? tb.phig + (s * 2 + g) * B : tb.phi + s * B, val);
            Vec<T, VEC> o;
#pragma unroll
            for (int u = 0; u < VEC; ++u) o.v[u] = val[u];
            stv<T, VEC>(FX + two_row<B>(rows, two, other, g) * nv + k, o);
        }
    }
    if constexpr (TWO) return;
    normal_velocity<T, VEC>(v1, v2, tab_load<SM>(fs), tab_load<SM>(fs + 1), vn);
    bool any = boundary;
#pragma unroll
    for (int u = 0; u < VEC; ++u) any = any || leaves(vn[u]);
    if (!any) return;
    point_value<T, VEC, B, SM>(fi, c, phi, val);
    const bool flux = sizeof(T) == 8 && !((meta & kFvSplitFlag) && (__ldg(ix.two + s) & kFvSplit));
    put_upwind<T, VEC>(FX + (int64_t)fid * nv + k, vn, val, other, boundary, flux);
}

// Pass 1 of one cell, any polygon.
template <typename T, int VEC, int MAXF, int B, int K, bool TWO>
__device__ __forceinline__ void recon_faces(const T *__restrict__ f, T *__restrict__ FX, const FvTables<T> &tb,
                                            const FvIdx &ix, int64_t rows, int64_t p, int ncf, int meta, int k, int nv,
                                            T v1, const T (&v2)[VEC], const Vec<T, VEC> &fi) {
    T c[B][VEC];
    if constexpr (sizeof(T) == 8) {
        static_assert(VEC == 1, "FP64 takes one velocity per thread");
        double c1[B];
        recon_coefs_f64<MAXF, B, K>(f, tb, ix, p, ncf, k, nv, fi.v[0], c1);
#pragma unroll
        for (int l = 0; l < B; ++l) c[l][0] = c1[l];
    } else {
        recon_coefs_f32<VEC, MAXF>(f, tb, ix, p, ncf, k, nv, fi, c);
    }
    const int nf = meta & 0xf;
#pragma unroll
    for (int q = 0; q < MAXF; ++q)
        if (q < nf)
            emit_face<T, VEC, B, false, TWO>(FX, tb, ix, rows, p, q, __ldg(ix.fid + p * kFvMaxFaces + q), meta, k, nv, v1,
                                             v2, fi, c, tb.fs + 2 * (p * kFvMaxFaces + q), tb.phi + (p * kFvMaxFaces + q) * B);
}

// Weights of one pair of velocities of a flagged triangle (kFvRegular: its
// stencil starts with the face neighbours; sector s joins faces s and s + 1
// mod 3) in FP32x2: c holds p_opt's coefficients, d the differences to the face
// neighbours; the steps of recon_coefs_f32.
template <int B>
__device__ __forceinline__ void weigh_tri(float2 (&c)[B], const float2 (&d)[3], const float4 (&R)[3],
                                          const float4 &quad) {
    constexpr float kLam0 = 0.75f, kInvLam0 = (float)(4.0 / 3.0), kEps = 1e-14f;
    const float lamL = 0.25f / 3.0f;
    float2 sx[3], sy[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const float2 da = d[s], db = d[(s + 1) % 3];
        sx[s] = fma2(dup2(R[s].x), da, mul2(dup2(R[s].y), db));
        sy[s] = fma2(dup2(R[s].z), da, mul2(dup2(R[s].w), db));
    }
    const float2 sumx = add2(add2(sx[0], sx[1]), sx[2]), sumy = add2(add2(sy[0], sy[1]), sy[2]);
    float2 p0[B];
    p0[0] = mul2(fma2(dup2(-lamL), sumx, c[0]), dup2(kInvLam0));
    p0[1] = mul2(fma2(dup2(-lamL), sumy, c[1]), dup2(kInvLam0));
#pragma unroll
    for (int l = 2; l < B; ++l) p0[l] = mul2(c[l], dup2(kInvLam0));
    float2 sig0 = fma2(p0[0], p0[0], mul2(p0[1], p0[1]));
    if constexpr (B == kFvCoef3) {
        const float2 A22 = dup2(4.f * quad.x + 4.f), A33 = dup2(quad.z + quad.x + 1.f), A44 = dup2(4.f * quad.z + 4.f);
        const float2 A23 = dup2(4.f * quad.y);
        sig0 = fma2(mul2(A22, p0[2]), p0[2], sig0);
        sig0 = fma2(mul2(A33, p0[3]), p0[3], sig0);
        sig0 = fma2(mul2(A44, p0[4]), p0[4], sig0);
        sig0 = fma2(mul2(A23, p0[2]), p0[3], sig0);
        sig0 = fma2(mul2(A23, p0[3]), p0[4], sig0);
    } else {
        sig0 = mul2(dup2(quad.w), sig0);
    }
    const float2 E = dup2(kEps);
    float2 sig[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        sig[s] = fma2(sx[s], sx[s], mul2(sy[s], sy[s]));
        if (B == 2) sig[s] = mul2(dup2(quad.w), sig[s]);
    }
    const float2 smin = make_float2(fminf(fminf(sig0.x, sig[0].x), fminf(sig[1].x, sig[2].x)),
                                    fminf(fminf(sig0.y, sig[0].y), fminf(sig[1].y, sig[2].y)));
    const float2 num = add2(smin, E);
    float2 r = mul2(num, rcp2(add2(sig0, E)));
    r = mul2(r, r);
    float2 w = mul2(dup2(kLam0), mul2(r, r)), wsum = w;
#pragma unroll
    for (int l = 0; l < B; ++l) p0[l] = mul2(w, p0[l]);
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        r = mul2(num, rcp2(add2(sig[s], E)));
        r = mul2(r, r);
        w = mul2(dup2(lamL), mul2(r, r));
        wsum = add2(wsum, w);
        p0[0] = fma2(w, sx[s], p0[0]);
        p0[1] = fma2(w, sy[s], p0[1]);
    }
    const float2 iw = rcp2(wsum);
#pragma unroll
    for (int l = 0; l < B; ++l) c[l] = mul2(p0[l], iw);
}

// Coefficients of the 4 velocities of a thread on a flagged triangle: row(q)
// gives f of stencil cell q, each row read once; then rows_read() is called.
// Rc, Rs, qd: the cell's table values.
template <int B, int K, bool SM, typename Row, typename Done>
__device__ __forceinline__ void coefs_tri_x2(const float *Rc, const float *Rs, const float *qd, const Vec<float, 4> &fi,
                                             Row row, Done rows_read, float (&c)[B][4]) {
    const float2 nf[2] = {make_float2(-fi.v[0], -fi.v[1]), make_float2(-fi.v[2], -fi.v[3])};
    float2 c2[2][B], dface[2][3];
#pragma unroll
    for (int q = 0; q < K; ++q) {
        const float4 r = row(q);
        const float2 d0 = add2(lo2(r), nf[0]), d1 = add2(hi2(r), nf[1]);
        if (q < 3) {
            dface[0][q] = d0;
            dface[1][q] = d1;
        }
#pragma unroll
        for (int l = 0; l < B; ++l) {
            const float2 R = dup2(tab_load<SM>(Rc + l * K + q));
            c2[0][l] = q == 0 ? mul2(R, d0) : fma2(R, d0, c2[0][l]);
            c2[1][l] = q == 0 ? mul2(R, d1) : fma2(R, d1, c2[1][l]);
        }
    }
    rows_read();
    float4 R[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) R[s] = tab_load<SM>(reinterpret_cast<const float4 *>(Rs + 4 * s));
    const float4 quad = tab_load<SM>(reinterpret_cast<const float4 *>(qd));
#pragma unroll
    for (int h = 0; h < 2; ++h) weigh_tri<B>(c2[h], dface[h], R, quad);
#pragma unroll
    for (int l = 0; l < B; ++l) {
        c[l][0] = c2[0][l].x;
        c[l][1] = c2[0][l].y;
        c[l][2] = c2[1][l].x;
        c[l][3] = c2[1][l].y;
    }
}

template <typename T, int VEC> struct Velocity {
    T v1, v2[VEC];
    __device__ __forceinline__ Velocity(int k, int N, T Lv, T dv) {
        const int j1 = k / N, j2 = k - j1 * N;
        v1 = -Lv + (T)j1 * dv;
#pragma unroll
        for (int u = 0; u < VEC; ++u) v2[u] = -Lv + (T)(j2 + u) * dv;
    }
};

// The nodes of VEC consecutive velocities, the two of a pair (N is even) in one
// row.  k / N by a product: k < 2^12 and N <= 64, so (k + 1/2) / N lies further
// from a whole number than FP32 rounds it.
template <typename T, int VEC> struct PairVelocity {
    T v1[(VEC + 1) / 2], v2[VEC];
    __device__ __forceinline__ PairVelocity(int k, int N, float iN, T Lv, T dv) {
        float j1 = floorf(((float)k + 0.5f) * iN), j2 = fmaf(-j1, (float)N, (float)k);
#pragma unroll
        for (int u = 0; u < VEC; ++u) {
            if (u > 0 && u % 2 == 0 && j2 + u >= (float)N) {
                j1 += 1.f;
                j2 -= (float)N;
            }
            if (u % 2 == 0) v1[u / 2] = fma((T)j1, dv, -Lv);
            v2[u] = fma((T)(j2 + u), dv, -Lv);
        }
    }
    // acc += v.n x
    __device__ __forceinline__ void add_flux(const typename C2<T>::type &n, const Vec<T, VEC> &x,
                                             Vec<T, VEC> &acc) const {
        if constexpr (sizeof(T) == 4 && VEC == 4) {
#pragma unroll
            for (int u = 0; u < 4; u += 2) {
                const float2 vn = fma2(make_float2(v2[u], v2[u + 1]), dup2(n.y), dup2(v1[u / 2] * n.x));
                const float2 a = fma2(vn, make_float2(x.v[u], x.v[u + 1]), make_float2(acc.v[u], acc.v[u + 1]));
                acc.v[u] = a.x;
                acc.v[u + 1] = a.y;
            }
        } else {
#pragma unroll
            for (int u = 0; u < VEC; ++u) acc.v[u] = fma(fma(v2[u], n.y, v1[u / 2] * n.x), x.v[u], acc.v[u]);
        }
    }
};

template <typename T, int VEC, int MAXF, int B, int K, bool TWO>
__device__ __forceinline__ void faces_block(const T *__restrict__ f, T *__restrict__ FX, const FvTables<T> &tb,
                                            const FvIdx &ix, int64_t rows, int nv, int N, T Lv, T dv) {
    griddep_launch();
    const int64_t p = blockIdx.x;
    const int k = (blockIdx.y * blockDim.x + threadIdx.x) * VEC;
    if (k >= nv) return;
    const int ncf = __ldg(ix.ncen + p), meta = __ldg(ix.meta + p);
    const Vec<T, VEC> fi = ldv<T, VEC>(f + (int64_t)__ldg(ix.order + p) * nv + k);
    const Velocity<T, VEC> v(k, N, Lv, dv);
    if constexpr (sizeof(T) == 4 && VEC == 4 && MAXF == 3) {
        if (ncf & kFvRegular) {      // uniform over the block: one cell per block
            float c[B][4];
            coefs_tri_x2<B, K, false>(tb.Rc + p * (B * K), tb.Rs + p * kFvMaxFaces * 4, tb.quad + 4 * p, fi, [&](int q) {
                return *reinterpret_cast<const float4 *>(f + (int64_t)__ldg(ix.cen + p * K + q) * nv + k);
            }, [] {}, c);
#pragma unroll
            for (int q = 0; q < 3; ++q)
                emit_face<float, 4, B, false, TWO>(FX, tb, ix, rows, p, q, __ldg(ix.fid + p * kFvMaxFaces + q), meta, k, nv,
                                              v.v1, v.v2, fi, c, tb.fs + 2 * (p * kFvMaxFaces + q),
                                              tb.phi + (p * kFvMaxFaces + q) * B);
            return;
        }
    }
    recon_faces<T, VEC, MAXF, B, K, TWO>(f, FX, tb, ix, rows, p, ncf, meta, k, nv, v.v1, v.v2, fi);
}

template <typename T, int VEC, int MAXF, int B, int K, bool TWO = false>
__global__ void __launch_bounds__(kFvThreads)
fv_faces_kernel(const T *__restrict__ f, T *__restrict__ FX, FvTables<T> tb, FvIdx ix, int64_t rows, int nv, int N, T Lv,
                T dv) {
    faces_block<T, VEC, MAXF, B, K, TWO>(f, FX, tb, ix, rows, nv, N, Lv, dv);
}

// Degree 2 on FP32 triangles with 4 | N, a block per cell (see faces3_launch).
// Bound by latency: four blocks of 256 threads per SM (64 registers, 36 bytes
// spilled) before three without spills, 16.5 and 18.5 us of a transport call on
// 409 cells x 32^2.
template <int BT, bool TWO>
__global__ void __launch_bounds__(BT, 4 * kFvThreads / BT)
fv_faces3_cell_kernel(const float *__restrict__ f, float *__restrict__ FX, FvTables<float> tb, FvIdx ix, int64_t rows,
                      int nv, int N, float Lv, float dv) {
    faces_block<float, 4, 3, kFvCoef3, kFvCentral3, TWO>(f, FX, tb, ix, rows, nv, N, Lv, dv);
}

// Degree 1 on FP32 triangles without walls: the same two passes with a cell's
// value at each of its faces, FV [cell][3][nv], in place of the upwind flux.
// Both passes are persistent: a block takes one of every (SMs x blocks per SM)
// positions of the processing order, walking them in steps of the grid; while
// it computes one cell, the rows of the next one travel into shared memory by
// cp.async (16 bytes per thread and row, each thread copying exactly the slots
// it reads back, so no block barrier is needed and warps past nv leave at
// once), and the index records of the cell after that are already being
// loaded.  Writing whole rows of values unmasked costs this light
// reconstruction less than forming and masking fluxes: 19802 triangles x 32^2,
// 0.094 + 0.055 ms (0.109 + 0.057 with table values loaded where they are
// used) against 0.137 + 0.050 ms with upwind flux rows.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_prev() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// The table values of a cell travel the same way, 4 bytes per lane into a buffer
// of the warp (read in the order of processing they come from DRAM, and a block
// that loads them when it needs them waits at every cell).
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}

constexpr int kFaceRows = 6;         // rows staged per cell: f_i and 5 stencil rows / 3 own and 3 neighbour face rows
// blocks per SM: 3 for the reconstruction (85 registers, no spills; 4 spill
// its record prefetch), 4 for the flux pass (64 registers)
constexpr int kFacesCtasPerSm = 3, kFluxCtasPerSm = 4;
// staged rows, then the warps' table values: 50 KB for 256 threads
constexpr size_t face_stage_bytes(int threads) {
    return 2 * kFaceRows * threads * sizeof(float4) + 2 * threads * sizeof(float);
}

// Degree 2 on FP32 triangles, the staged form for large meshes (see
// faces3_launch): pass 1 persistent in the same way, with the 12 rows of a
// stencil, the cell's table values and its indices staged, the indices one cell
// further ahead, per warp.  The rows have one buffer: the next cell's are asked
// for as soon as the differences have been formed, and arrive while this one's
// weights and faces are computed.  Blocks per SM: two of 256 threads (58 KB each,
// 128 registers a thread), as many warps as three such with narrower ones.
constexpr int kRows3 = 1 + kFvCentral3;
constexpr int kTab3Rs = 0, kTab3Quad = 12, kTab3Rc = 16, kTab3Phi = 71, kTab3Fs = 86, kTab3Values = 92;
constexpr int kIdx3Cen = 0, kIdx3Fid = 11, kIdx3Order = 14, kIdx3Meta = 15, kIdx3Ncen = 16, kIdx3Values = 17;
constexpr int kTab3Pitch = 96, kIdx3Pitch = 20;   // per warp and buffer
constexpr size_t faces3_stage_bytes(int threads) {
    return kRows3 * threads * sizeof(float4) +
           threads / 32 * (2 * kTab3Pitch * sizeof(float) + 3 * kIdx3Pitch * sizeof(int));
}

constexpr int faces3_ctas_per_sm(int threads) { return threads < kFvThreads ? 3 : 2; }
template <int BT, bool TWO>
__global__ void __launch_bounds__(BT, faces3_ctas_per_sm(BT) * kFvThreads / BT)
fv_faces3_persist_kernel(const float *__restrict__ f, float *__restrict__ FX, FvTables<float> tb, FvIdx ix,
                         int64_t rows, int64_t n, int nv, int N, float Lv, float dv) {
    constexpr int B = kFvCoef3, K = kFvCentral3, W = BT / 32;
    extern __shared__ float4 stage[];            // [kRows3][BT], [2][W][kTab3Pitch], [3][W][kIdx3Pitch]
    griddep_launch();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int kt = (blockIdx.y * BT + t) * 4;
    if (kt - 4 * lane >= nv || (int64_t)blockIdx.x >= n) return;   // warps past nv
    const bool act = kt < nv;
    const int k = act ? kt : 0;                  // the last warp's idle lanes store nothing
    float *const tabs = reinterpret_cast<float *>(stage + kRows3 * BT) + warp * kTab3Pitch;
    int *const idxs = reinterpret_cast<int *>(reinterpret_cast<float *>(stage + kRows3 * BT) + 2 * W * kTab3Pitch) +
                      warp * kIdx3Pitch;
    const int64_t G = gridDim.x;
    // this lane's index word, and its three table values, of position 0 and the distances between positions
    const int *is = lane < kIdx3Fid ? ix.cen + lane : lane < kIdx3Order ? ix.fid + (lane - kIdx3Fid)
                  : lane == kIdx3Order ? ix.order : lane == kIdx3Meta ? ix.meta : ix.ncen;
    const int id = lane < kIdx3Fid ? K : lane < kIdx3Order ? kFvMaxFaces : 1;
    const float *ts[3];
    int td[3];
#pragma unroll
    for (int u = 0; u < 3; ++u) {
        const int e = lane + 32 * u;
        ts[u] = e < kTab3Quad ? tb.Rs + e : e < kTab3Rc ? tb.quad + (e - kTab3Quad) : e < kTab3Phi ? tb.Rc + (e - kTab3Rc)
              : e < kTab3Fs ? tb.phi + (e - kTab3Phi) : tb.fs + (e - kTab3Fs);
        td[u] = e < kTab3Quad ? kFvMaxFaces * 4 : e < kTab3Rc ? 4 : e < kTab3Phi ? B * K
              : e < kTab3Fs ? kFvMaxFaces * B : kFvMaxFaces * 2;
    }
    auto issue_idx = [&](int64_t pr, int slot) {
        if (lane < kIdx3Values) cp_async4(idxs + slot * W * kIdx3Pitch + lane, is + pr * id);
    };
    float4 *const sl = stage + t;
    auto issue = [&](int64_t pr, int slot, int buf) {
#pragma unroll
        for (int u = 0; u < 3; ++u)
            if (lane + 32 * u < kTab3Values) cp_async4(tabs + buf * W * kTab3Pitch + lane + 32 * u, ts[u] + pr * td[u]);
        const int *x = idxs + slot * W * kIdx3Pitch;
        cp_async16(sl, f + (int64_t)x[kIdx3Order] * nv + k);
#pragma unroll
        for (int q = 0; q < K; ++q)              // a short stencil's other entries are cell 0
            cp_async16(sl + (q + 1) * BT, f + (int64_t)x[kIdx3Cen + q] * nv + k);
    };
    const Velocity<float, 4> v(k, N, Lv, dv);
    int64_t p = blockIdx.x;
    issue_idx(p, 0);
    cp_async_commit();
    cp_async_wait_all();
    __syncwarp();
    issue(p, 0, 0);
    if (p + G < n) issue_idx(p + G, 1);
    cp_async_commit();
    int slot = 0;
    for (int it = 0;; ++it) {
        const bool more = p + G < n;
        const int next = slot == 2 ? 0 : slot + 1, after = next == 2 ? 0 : next + 1;
        cp_async_wait_all();
        __syncwarp();
        auto ahead = [&] {
            if (more) issue(p + G, next, (it + 1) & 1);
            if (p + 2 * G < n) issue_idx(p + 2 * G, after);
            cp_async_commit();
        };
        const int *x = idxs + slot * W * kIdx3Pitch;
        const float *tab = tabs + (it & 1) * W * kTab3Pitch;
        const int meta = x[kIdx3Meta], ncf = x[kIdx3Ncen];
        Vec<float, 4> fi;
        const float4 f4 = sl[0];
        fi.v[0] = f4.x; fi.v[1] = f4.y; fi.v[2] = f4.z; fi.v[3] = f4.w;
        if (ncf & kFvRegular) {
            float c[B][4];
            coefs_tri_x2<B, K, true>(tab + kTab3Rc, tab + kTab3Rs, tab + kTab3Quad, fi,
                                     [&](int q) { return sl[(q + 1) * BT]; }, ahead, c);
#pragma unroll
            for (int q = 0; act && q < 3; ++q)
                emit_face<float, 4, B, true, TWO>(FX, tb, ix, rows, p, q, x[kIdx3Fid + q], meta, k, nv, v.v1, v.v2, fi, c,
                                             tab + kTab3Fs + 2 * q, tab + kTab3Phi + B * q);
        } else {
            ahead();
            if (act) recon_faces<float, 4, 3, B, K, TWO>(f, FX, tb, ix, rows, p, ncf, meta, k, nv, v.v1,
                                                    v.v2, fi);
        }
        if (!more) break;
        __syncwarp();
        p += G;
        slot = next;
    }
}

// CWENO gradient of one pair of velocities of a flagged triangle (kFvRegular):
// d[q] = fbar_{cen q} - fbar_i, the face neighbours in d[0..2]; sector s
// joins faces s and s + 1 mod 3.  The steps are those of
// recon_coefs_f32 (central gradient, sector gradients, g_0, smoothness, weights as
// lambda_s ((sigma_min + eps) / (sigma_s + eps))^4, normalised sum).
__device__ __forceinline__ void cweno_pair_tri(const float2 (&d)[kFvCentral], const float (&rx)[kFvCentral],
                                               const float (&ry)[kFvCentral], const float4 (&R)[3], float h2,
                                               float2 &gx_out, float2 &gy_out) {
    constexpr float kLam0 = 0.75f, kInvLam0 = (float)(4.0 / 3.0), kEps = 1e-14f;
    const float lamL = 0.25f / 3.0f;
    float2 gx = mul2(dup2(rx[0]), d[0]), gy = mul2(dup2(ry[0]), d[0]);
#pragma unroll
    for (int q = 1; q < kFvCentral; ++q) {
        gx = fma2(dup2(rx[q]), d[q], gx);
        gy = fma2(dup2(ry[q]), d[q], gy);
    }
    float2 sx[3], sy[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const float2 da = d[s], db = d[(s + 1) % 3];
        sx[s] = fma2(dup2(R[s].x), da, mul2(dup2(R[s].y), db));
        sy[s] = fma2(dup2(R[s].z), da, mul2(dup2(R[s].w), db));
    }
    const float2 sumx = add2(add2(sx[0], sx[1]), sx[2]), sumy = add2(add2(sy[0], sy[1]), sy[2]);
    const float2 g0x = mul2(fma2(dup2(-lamL), sumx, gx), dup2(kInvLam0));
    const float2 g0y = mul2(fma2(dup2(-lamL), sumy, gy), dup2(kInvLam0));
    const float2 H = dup2(h2), E = dup2(kEps);
    const float2 sig0 = mul2(H, fma2(g0x, g0x, mul2(g0y, g0y)));
    float2 sig[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) sig[s] = mul2(H, fma2(sx[s], sx[s], mul2(sy[s], sy[s])));
    const float2 smin = make_float2(fminf(fminf(sig0.x, sig[0].x), fminf(sig[1].x, sig[2].x)),
                                    fminf(fminf(sig0.y, sig[0].y), fminf(sig[1].y, sig[2].y)));
    const float2 num = add2(smin, E);
    float2 r = mul2(num, rcp2(add2(sig0, E)));
    r = mul2(r, r);
    float2 w = mul2(dup2(kLam0), mul2(r, r));
    float2 wsum = w, ax = mul2(w, g0x), ay = mul2(w, g0y);
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        r = mul2(num, rcp2(add2(sig[s], E)));
        r = mul2(r, r);
        w = mul2(dup2(lamL), mul2(r, r));
        wsum = add2(wsum, w);
        ax = fma2(w, sx[s], ax);
        ay = fma2(w, sy[s], ay);
    }
    const float2 iw = rcp2(wsum);
    gx_out = mul2(ax, iw);
    gy_out = mul2(ay, iw);
}

// Values at the three faces of the 4 velocities k..k+3 of a flagged triangle;
// tab: its table values (kTabRs ...).
constexpr int kTabRs = 0, kTabRc = 12, kTabPhi = 22, kTabH2 = 28, kTabValues = 29;
__device__ __forceinline__ void tri_values_x2(float *__restrict__ FV, const float *tab, const float4 (&fr)[kFvCentral],
                                              int64_t i, int k, int nv, const float4 fi, bool act) {
    float rx[kFvCentral], ry[kFvCentral];
#pragma unroll
    for (int q = 0; q < kFvCentral; ++q) {
        rx[q] = tab[kTabRc + q];
        ry[q] = tab[kTabRc + kFvCentral + q];
    }
    float4 R[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) R[s] = *reinterpret_cast<const float4 *>(tab + kTabRs + 4 * s);
    const float h2 = tab[kTabH2];
    float2 gx[2], gy[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float2 nf = neg2(h == 0 ? lo2(fi) : hi2(fi));
        float2 d[kFvCentral];
#pragma unroll
        for (int q = 0; q < kFvCentral; ++q) d[q] = add2(h == 0 ? lo2(fr[q]) : hi2(fr[q]), nf);
        cweno_pair_tri(d, rx, ry, R, h2, gx[h], gy[h]);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float2 ox = dup2(tab[kTabPhi + 2 * q]), oy = dup2(tab[kTabPhi + 2 * q + 1]);
        const float2 a = fma2(gy[0], oy, fma2(gx[0], ox, lo2(fi)));
        const float2 b = fma2(gy[1], oy, fma2(gx[1], ox, hi2(fi)));
        if (act) *reinterpret_cast<float4 *>(FV + (i * 3 + q) * nv + k) = make_float4(a.x, a.y, b.x, b.y);
    }
}

// Index record of position p needed by the reconstruction: cell, flags, stencil.
struct RecG {
    int i, ncf, c[kFvCentral];
};
__device__ __forceinline__ RecG rec_g(const int4 *__restrict__ tripos, int64_t p) {
    const int4 a = __ldg(tripos + 3 * p), b = __ldg(tripos + 3 * p + 1), c = __ldg(tripos + 3 * p + 2);
    return RecG{a.x, a.y, {b.x, b.y, b.z, b.w, c.x}};
}

template <int BT>
__global__ void __launch_bounds__(BT, kFacesCtasPerSm * kFvThreads / BT)
fv_values_persist_kernel(const float *__restrict__ f, float *__restrict__ FV, FvTables<float> tb, FvIdx ix,
                         const int4 *__restrict__ tripos, int64_t n, int nv) {
    extern __shared__ float4 stage[];            // [2][kFaceRows][BT], [2][warp][32] table values
    griddep_launch();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    float *const tabs = reinterpret_cast<float *>(stage + 2 * kFaceRows * BT) + warp * 32;
    const int kt = (blockIdx.y * BT + t) * 4;
    if (kt - 4 * lane >= nv || (int64_t)blockIdx.x >= n) return;   // warps past nv
    const bool act = kt < nv;
    const int k = act ? kt : 0;                  // the last warp's idle lanes store nothing
    const int64_t G = gridDim.x;
    // this lane's table value of position 0, and the distance between positions
    const float *ts = lane < kTabRc ? tb.Rs + lane : lane < kTabPhi ? tb.Rc + (lane - kTabRc)
                    : lane < kTabH2 ? tb.phi + (lane - kTabPhi) : tb.quad + 3;
    const int td = lane < kTabRc ? kFvMaxFaces * 4 : lane < kTabPhi ? 2 * kFvCentral : lane < kTabH2 ? 2 * kFvMaxFaces : 4;
    auto issue = [&](const RecG &r, int64_t pr, int buf) {
        if (lane < kTabValues) cp_async4(tabs + buf * BT + lane, ts + pr * td);
        float4 *sl = stage + buf * kFaceRows * BT + t;
        cp_async16(sl, f + (int64_t)r.i * nv + k);
#pragma unroll
        for (int q = 0; q < kFvCentral; ++q) cp_async16(sl + (q + 1) * BT, f + (int64_t)r.c[q] * nv + k);
    };
    int64_t p = blockIdx.x;
    RecG cur = rec_g(tripos, p);
    issue(cur, p, 0);
    cp_async_commit();
    RecG nxt = cur;
    if (p + G < n) nxt = rec_g(tripos, p + G);
    for (int it = 0;; ++it) {
        const bool more = p + G < n;
        if (more) issue(nxt, p + G, (it + 1) & 1);
        cp_async_commit();
        RecG nn = nxt;
        if (p + 2 * G < n) nn = rec_g(tripos, p + 2 * G);
        cp_async_wait_prev();
        __syncwarp();
        const float4 *sl = stage + (it & 1) * kFaceRows * BT + t;
        const float4 fi = sl[0];
        if (cur.ncf & kFvRegular) {
            float4 fr[kFvCentral];
#pragma unroll
            for (int q = 0; q < kFvCentral; ++q) fr[q] = sl[(q + 1) * BT];
            tri_values_x2(FV, tabs + (it & 1) * BT, fr, cur.i, k, nv, fi, act);
        } else {
            Vec<float, 4> fv;
            fv.v[0] = fi.x; fv.v[1] = fi.y; fv.v[2] = fi.z; fv.v[3] = fi.w;
            float c[2][4], val[4];
            recon_coefs_f32<4, 3>(f, tb, ix, p, cur.ncf, k, nv, fv, c);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                point_value<float, 4, 2>(fv, c, tb.phi + (p * kFvMaxFaces + q) * 2, val);
                if (act)
                    *reinterpret_cast<float4 *>(FV + ((int64_t)cur.i * 3 + q) * nv + k) =
                        make_float4(val[0], val[1], val[2], val[3]);
            }
        }
        if (!more) break;
        __syncwarp();
        p += G;
        cur = nxt;
        nxt = nn;
    }
}

// Index record of position p needed by the flux pass: cell, neighbours, their face indices.
struct RecF {
    int i, qbits, nb[3];
};
__device__ __forceinline__ RecF rec_f(const int4 *__restrict__ tripos, int64_t p) {
    const int4 a = __ldg(tripos + 3 * p), c = __ldg(tripos + 3 * p + 2);
    return RecF{a.x, a.w, {c.y, c.z, c.w}};
}

template <int BT>
__global__ void __launch_bounds__(BT, kFluxCtasPerSm * kFvThreads / BT)
fv_flux_values_persist_kernel(const float *FV, float *__restrict__ L, FvTables<float> tb,
                             const int4 *__restrict__ tripos, int64_t n, int nv, int N, float Lv, float dv) {
    extern __shared__ float4 stage[];            // [2][kFaceRows][BT], [2][warp][32]: 3 (nx, ny), 1 / area
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    float *const tabs = reinterpret_cast<float *>(stage + 2 * kFaceRows * BT) + warp * 32;
    const int kt = (blockIdx.y * BT + t) * 4;
    if (kt - 4 * lane >= nv || (int64_t)blockIdx.x >= n) return;
    const bool act = kt < nv;
    const int k = act ? kt : 0;
    const int64_t G = gridDim.x;
    // positions from the end of the order (the rows the reconstruction wrote last are still in L2)
    auto pos = [&](int64_t p) { return n - 1 - p; };
    auto issue = [&](const RecF &r, int64_t pr, int buf) {
        if (lane < 7)
            cp_async4(tabs + buf * BT + lane, lane < 6 ? tb.fn + pos(pr) * kFvMaxFaces * 2 + lane : tb.inv_area + pos(pr));
        float4 *sl = stage + buf * kFaceRows * BT + t;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            cp_async16(sl + q * BT, FV + ((int64_t)r.i * 3 + q) * nv + k);
            if (r.nb[q] >= 0)
                cp_async16(sl + (3 + q) * BT, FV + ((int64_t)r.nb[q] * 3 + ((r.qbits >> (2 * q)) & 3)) * nv + k);
        }
    };
    const int j1 = k / N, j2 = k - j1 * N;
    const float v1 = -Lv + (float)j1 * dv;
    float2 v2[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) v2[h] = make_float2(-Lv + (float)(j2 + 2 * h) * dv, -Lv + (float)(j2 + 2 * h + 1) * dv);
    const float2 hf = dup2(0.5f);
    int64_t p = blockIdx.x;
    RecF cur = rec_f(tripos, pos(p));
    griddep_wait();                              // launched while the reconstruction ends
    issue(cur, p, 0);
    cp_async_commit();
    RecF nxt = cur;
    if (p + G < n) nxt = rec_f(tripos, pos(p + G));
    for (int it = 0;; ++it) {
        const bool more = p + G < n;
        if (more) issue(nxt, p + G, (it + 1) & 1);
        cp_async_commit();
        RecF nn = nxt;
        if (p + 2 * G < n) nn = rec_f(tripos, pos(p + 2 * G));
        cp_async_wait_prev();
        __syncwarp();
        const float *tab = tabs + (it & 1) * BT;
        const float4 *sl = stage + (it & 1) * kFaceRows * BT + t;
        const int64_t i = cur.i;
        float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float4 fl = sl[q * BT];
            const float4 fr = cur.nb[q] >= 0 ? sl[(3 + q) * BT] : fl;
            const float nx = tab[2 * q], ny = tab[2 * q + 1];
            const float2 v1nx = dup2(v1 * nx);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 a = h == 0 ? lo2(fl) : hi2(fl), b = h == 0 ? lo2(fr) : hi2(fr);
                const float2 vn = fma2(v2[h], dup2(ny), v1nx);
                const float2 hv = mul2(hf, vn), nah = make_float2(-fabsf(hv.x), -fabsf(hv.y));
                acc[h] = fma2(hv, add2(a, b), acc[h]);
                acc[h] = fma2(nah, add2(b, make_float2(-a.x, -a.y)), acc[h]);
            }
        }
        const float2 ia = dup2(tab[6]);
        const float2 o0 = mul2(acc[0], ia), o1 = mul2(acc[1], ia);
        if (act) *reinterpret_cast<float4 *>(L + i * nv + k) = make_float4(o0.x, o0.y, o1.x, o1.y);
        if (!more) break;
        __syncwarp();
        p += G;
        cur = nxt;
        nxt = nn;
    }
}

// Incoming half of a wall face (full accommodation, eq. BOU with alpha = 1,
// eq. MAXB, eq. MU): one block per wall holds all nv <= 1024 velocities, 4 per
// thread.  mu, the ratio of the outgoing mass flux sum_{v.n > 0} f_L v.n (the
// face row as pass 1 wrote it; FP32: times v.n) to the incoming flux of the unit
// wall Maxwellian sum_{v.n < 0} M_w |v.n|, is a block reduction (FP64, fixed
// order); velocities entering the domain get mu M_w(v) (FP64: times v.n).  For
// degree 2 the balance at the face's two Gauss points is linear in the
// outgoing flux, so the mean over the face is balanced once.
template <typename T>
__global__ void __launch_bounds__(kFvThreads)
fv_wall_faces_kernel(T *__restrict__ FX, FvTables<T> tb, const int *__restrict__ fid, const int *__restrict__ wall,
                     const int64_t *__restrict__ wallslot, const T *__restrict__ wallp, int nv, int N, T Lv, T dv) {
    constexpr bool FLUX = sizeof(T) == 8;
    __shared__ double red[2 * (kFvThreads / 32)];
    const int w = blockIdx.x;
    const int64_t s = wallslot[w];
    if (wall[s] != w) return;                    // an edge named twice: the last wall holds
    const int kt = threadIdx.x * 4;
    const bool act = kt < nv;
    const int k = act ? kt : 0;                  // idle threads store nothing
    T *row = FX + (int64_t)__ldg(fid + s) * nv + k;
    const Velocity<T, 4> v(k, N, Lv, dv);
    T vn[4], mw[4];
    normal_velocity<T, 4>(v.v1, v.v2, __ldg(tb.fn + 2 * s), __ldg(tb.fn + 2 * s + 1), vn);
    const T th = __ldg(wallp + 3 * w), uw1 = __ldg(wallp + 3 * w + 1), uw2 = __ldg(wallp + 3 * w + 2);
    const T inv2th = (T)0.5 / th, norm = (T)(0.15915494309189535) / th;   // 1 / (2 pi theta)
    double num = 0.0, den = 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const T d1 = v.v1 - uw1, d2 = v.v2[u] - uw2;
        mw[u] = norm * exp(-(d1 * d1 + d2 * d2) * inv2th);
        if (act && vn[u] > (T)0) num += (double)(FLUX ? row[u] : row[u] * vn[u]);
        if (act && vn[u] < (T)0) den += (double)(mw[u] * -vn[u]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        num += __shfl_xor_sync(0xffffffffu, num, o);
        den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[2 * (threadIdx.x >> 5)] = num;
        red[2 * (threadIdx.x >> 5) + 1] = den;
    }
    __syncthreads();
    num = den = 0.0;
#pragma unroll
    for (int q = 0; q < kFvThreads / 32; ++q) {
        num += red[2 * q];
        den += red[2 * q + 1];
    }
    const T mu = (T)(num / den);
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (act && !(vn[u] > (T)0)) row[u] = FLUX ? vn[u] * (mu * mw[u]) : mu * mw[u];
}

// Pass 2: L_i = (1/|P_i|) sum over the faces of v.n times their rows (FP64: of the
// signed rows), the cells in the reverse of pass 1's order, so that the first ones
// find the rows written last still in L2.  DRAM-bound, and by latency: every
// table value is asked for before the rows, and 32 registers keep the SMs full, so
// the thin cells' branch forms its velocities anew (19802 triangles x 32^2, FP32:
// 49.5 us; 69 us with the normals loaded where they are used, 56 with 40
// registers, 53 with the velocities kept, which spills).
template <typename T, int VEC, int MAXF, int B>
__global__ void __launch_bounds__(kFvThreads, MAXF == 3 ? 8 : 4)
fv_sum_kernel(const T *FX, T *__restrict__ L, FvTables<T> tb, FvIdx ix, const int *__restrict__ wall,
              int64_t rows, int nv, int N, float iN, T Lv, T dv) {
    constexpr bool F64 = sizeof(T) == 8;
    const int64_t p = gridDim.x - 1 - blockIdx.x;
    const int k = (blockIdx.y * kFvThreads + threadIdx.x) * VEC;
    if (k >= nv) return;
    using V2 = typename C2<T>::type;
    const V2 *fn = reinterpret_cast<const V2 *>(tb.fn) + p * kFvMaxFaces;
    // every table value before the wait: they come from DRAM, one latency for all
    const int meta = __ldg(ix.meta + p), nf = MAXF == 3 ? 3 : meta & 0xf;
    int row[MAXF];
    V2 n[MAXF];
#pragma unroll
    for (int q = 0; q < MAXF; ++q) {
        row[q] = __ldg(ix.fid + p * kFvMaxFaces + q);
        if constexpr (!F64) n[q] = __ldg(fn + q);
    }
    const T ia = __ldg(tb.inv_area + p);
    const int64_t i = __ldg(ix.order + p);
    auto velocity = [&] { return PairVelocity<T, VEC>(k, N, iN, Lv, dv); };
    griddep_wait();                      // launched while pass 1 ends: its rows from here on
    Vec<T, VEC> x[MAXF];
#pragma unroll
    for (int q = 0; q < MAXF; ++q)
        if (q < nf) x[q] = ldv_after<T, VEC>(FX + (int64_t)row[q] * nv + k);
    Vec<T, VEC> o;
#pragma unroll
    for (int u = 0; u < VEC; ++u) o.v[u] = (T)0;
    if constexpr (F64) {
        if (!(meta & kFvSplitFlag)) {
#pragma unroll
            for (int q = 0; q < MAXF; ++q) {
                if (q >= nf) continue;
                const bool other = (meta >> (8 + q)) & 1;
#pragma unroll
                for (int u = 0; u < VEC; ++u) o.v[u] += negate_if(other, x[q].v[u]);
            }
        } else {
            const PairVelocity<T, VEC> v = velocity();
#pragma unroll
            for (int q = 0; q < MAXF; ++q) {
                if (q >= nf) continue;
                const Vec<T, VEC> &y = x[q];
                if (__ldg(ix.two + p * kFvMaxFaces + q) & kFvSplit) {
                    v.add_flux(__ldg(fn + q), y, o);
                } else {
                    const bool other = (meta >> (8 + q)) & 1;
#pragma unroll
                    for (int u = 0; u < VEC; ++u) o.v[u] += negate_if(other, y.v[u]);
                }
            }
        }
    } else {
        const unsigned two_sided = (unsigned)meta >> 24;
        const PairVelocity<T, VEC> v = velocity();
#pragma unroll
        for (int q = 0; q < MAXF; ++q)
            if (q < nf && !((two_sided >> q) & 1)) v.add_flux(n[q], x[q], o);
        if (two_sided) {
            // faces of thin cells: (v.n)(f_L + f_R)/2 - |v.n| (f_R - f_L)/2 at every face point
            constexpr int GP = B == kFvCoef3 ? 2 : 1;
            constexpr T half = (T)(0.5 / GP);
#pragma unroll 1
            for (int q = 0; q < nf; ++q) {
                if (!((two_sided >> q) & 1)) continue;
                const int64_t s = p * kFvMaxFaces + q;
                const V2 nq = __ldg(fn + q);
                if (wall && __ldg(wall + s) >= 0) {          // the wall's row
                    v.add_flux(nq, ldv_after<T, VEC>(FX + (int64_t)__ldg(ix.fid + s) * nv + k), o);
                    continue;
                }
                const int side = (meta >> (8 + q)) & 1, two = __ldg(ix.two + s) & (kFvSplit - 1);
                const bool boundary = (meta >> (16 + q)) & 1;
#pragma unroll 1
                for (int g = 0; g < GP; ++g) {
                    const T *a = FX + two_row<B>(rows, two, side, g) * nv + k;
                    // the other side's points run the other way
                    const T *b = boundary ? a : FX + two_row<B>(rows, two, 1 - side, GP - 1 - g) * nv + k;
#pragma unroll
                    for (int u = 0; u < VEC; ++u) {
                        const PairVelocity<T, 1> w(k + u, N, iN, Lv, dv);
                        const T h = half * fma(w.v2[0], nq.y, w.v1[0] * nq.x), fl = __ldcg(a + u), fr = __ldcg(b + u);
                        o.v[u] = fma(h, fl + fr, o.v[u]);
                        o.v[u] = fma(-fabs(h), fr - fl, o.v[u]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int u = 0; u < VEC; ++u) o.v[u] *= ia;
    stv<T, VEC>(L + i * nv + k, o);
}

// Pass 2 where every face is two-sided (FP32, degree 2): the Rusanov form at
// both points of every face, term by term as in the two-sided faces above.
template <int VEC, int MAXF>
__global__ void __launch_bounds__(kFvThreads)
fv_sum_two_kernel(const float *FX, float *__restrict__ L, FvTables<float> tb, FvIdx ix, int nv, int N,
                  float Lv, float dv) {
    const int64_t p = gridDim.x - 1 - blockIdx.x;
    const int k = (blockIdx.y * kFvThreads + threadIdx.x) * VEC;
    if (k >= nv) return;
    const int meta = __ldg(ix.meta + p), nf = meta & 0xf;
    const Velocity<float, VEC> v(k, N, Lv, dv);
    const float ia = __ldg(tb.inv_area + p);
    griddep_wait();
    Vec<float, VEC> o;
#pragma unroll
    for (int u = 0; u < VEC; ++u) o.v[u] = 0.f;
#pragma unroll
    for (int q = 0; q < MAXF; ++q) {
        if (q >= nf) continue;
        const int64_t s = p * kFvMaxFaces + q;
        const int side = (meta >> (8 + q)) & 1, fid = __ldg(ix.fid + s);
        const bool boundary = (meta >> (16 + q)) & 1;
        float vn[VEC];
        normal_velocity<float, VEC>(v.v1, v.v2, __ldg(tb.fn + 2 * s), __ldg(tb.fn + 2 * s + 1), vn);
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const Vec<float, VEC> a = ldv_after<float, VEC>(FX + two_row<kFvCoef3>(0, fid, side, g) * nv + k);
            const Vec<float, VEC> b =
                boundary ? a : ldv_after<float, VEC>(FX + two_row<kFvCoef3>(0, fid, 1 - side, 1 - g) * nv + k);
#pragma unroll
            for (int u = 0; u < VEC; ++u) {
                const float h = 0.25f * vn[u];
                o.v[u] = fma(h, a.v[u] + b.v[u], o.v[u]);
                o.v[u] = fma(-fabsf(h), b.v[u] - a.v[u], o.v[u]);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < VEC; ++u) o.v[u] *= ia;
    stv<float, VEC>(L + (int64_t)__ldg(ix.order + p) * nv + k, o);
}

// ---- order 1: Rusanov fluxes of the cell averages in one pass ------------------
template <typename T, int VEC, int MAXF>
__global__ void __launch_bounds__(kFvThreads, (sizeof(T) == 4 && VEC == 4 && MAXF <= 3) ? 4 : 1)
fv_first_kernel(const T *__restrict__ f, T *__restrict__ L, FvTables<T> tb, FvIdx ix, const int *__restrict__ nb,
                int nv, int N, T Lv, T dv) {
    const int64_t p = blockIdx.x;
    const int k = (blockIdx.y * kFvThreads + threadIdx.x) * VEC;
    if (k >= nv) return;
    const int64_t i = __ldg(ix.order + p);
    const int nf = __ldg(ix.meta + p) & 0xf;
    const Vec<T, VEC> fi = ldv<T, VEC>(f + i * nv + k);
    // every face's neighbour row first
    Vec<T, VEC> fj[MAXF];
#pragma unroll
    for (int q = 0; q < MAXF; ++q) {
        const int j = q < nf ? __ldg(nb + p * kFvMaxFaces + q) : -1;
        fj[q] = fi;
        if (j >= 0) fj[q] = ldv<T, VEC>(f + (int64_t)j * nv + k);
    }
    const Velocity<T, VEC> v(k, N, Lv, dv);
    T acc[VEC];
#pragma unroll
    for (int u = 0; u < VEC; ++u) acc[u] = (T)0;
#pragma unroll
    for (int q = 0; q < MAXF; ++q) {
        if (q >= nf) continue;
        const int64_t s = p * kFvMaxFaces + q;
        T vn[VEC];
        normal_velocity<T, VEC>(v.v1, v.v2, __ldg(tb.fn + 2 * s), __ldg(tb.fn + 2 * s + 1), vn);
#pragma unroll
        for (int u = 0; u < VEC; ++u) {
            const T fl = fi.v[u], fr = fj[q].v[u];
            acc[u] += (T)0.5 * vn[u] * (fl + fr) - (T)0.5 * fabs(vn[u]) * (fr - fl);
        }
    }
    const T ia = __ldg(tb.inv_area + p);
    Vec<T, VEC> o;
#pragma unroll
    for (int u = 0; u < VEC; ++u) o.v[u] = acc[u] * ia;
    stv<T, VEC>(L + i * nv + k, o);
}

// Order 1 on a mesh with walls: one block holds all nv <= 1024 velocities of
// its cell, 4 per thread, and forms each wall face's mu as
// fv_wall_faces_kernel does.
template <typename T, int MAXF>
__global__ void __launch_bounds__(kFvThreads)
fv_first_wall_kernel(const T *__restrict__ f, T *__restrict__ L, FvTables<T> tb, FvIdx ix, const int *__restrict__ nb,
                     const int *__restrict__ wall, const T *__restrict__ wallp, int nv, int N, T Lv, T dv) {
    __shared__ double red[2 * (kFvThreads / 32)];
    const int64_t p = blockIdx.x, i = __ldg(ix.order + p);
    const int kt = threadIdx.x * 4;
    const bool act = kt < nv;
    const int k = act ? kt : 0;                  // idle threads read row 0 and store nothing
    const int nf = __ldg(ix.meta + p) & 0xf;
    const Vec<T, 4> fi = ld4<T>(f + i * nv + k);
    const Velocity<T, 4> v(k, N, Lv, dv);
    T acc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] = (T)0;
#pragma unroll
    for (int q = 0; q < MAXF; ++q) {
        if (q >= nf) continue;                   // uniform over the block (one cell)
        const int64_t s = p * kFvMaxFaces + q;
        const int j = __ldg(nb + s);
        T vn[4];
        normal_velocity<T, 4>(v.v1, v.v2, __ldg(tb.fn + 2 * s), __ldg(tb.fn + 2 * s + 1), vn);
        Vec<T, 4> fr = fi;
        if (j >= 0) fr = ld4<T>(f + (int64_t)j * nv + k);
        const int w = j < 0 ? __ldg(wall + s) : -1;          // uniform over the block
        if (w >= 0) {
            const T th = __ldg(wallp + 3 * w), uw1 = __ldg(wallp + 3 * w + 1), uw2 = __ldg(wallp + 3 * w + 2);
            const T inv2th = (T)0.5 / th, norm = (T)(0.15915494309189535) / th;   // 1 / (2 pi theta)
            T mw[4];
            double num = 0.0, den = 0.0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const T d1 = v.v1 - uw1, d2 = v.v2[u] - uw2;
                mw[u] = norm * exp(-(d1 * d1 + d2 * d2) * inv2th);
                if (act && vn[u] > (T)0) num += (double)(fi.v[u] * vn[u]);
                if (act && vn[u] < (T)0) den += (double)(mw[u] * -vn[u]);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                num += __shfl_xor_sync(0xffffffffu, num, o);
                den += __shfl_xor_sync(0xffffffffu, den, o);
            }
            __syncthreads();                     // red is reused face after face
            if ((threadIdx.x & 31) == 0) {
                red[2 * (threadIdx.x >> 5)] = num;
                red[2 * (threadIdx.x >> 5) + 1] = den;
            }
            __syncthreads();
            num = den = 0.0;
#pragma unroll
            for (int q2 = 0; q2 < kFvThreads / 32; ++q2) {
                num += red[2 * q2];
                den += red[2 * q2 + 1];
            }
            const T mu = (T)(num / den);
#pragma unroll
            for (int u = 0; u < 4; ++u) fr.v[u] = vn[u] > (T)0 ? fi.v[u] : mu * mw[u];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            acc[u] += (T)0.5 * vn[u] * (fi.v[u] + fr.v[u]) - (T)0.5 * fabs(vn[u]) * (fr.v[u] - fi.v[u]);
    }
    if (act) {
        const T ia = __ldg(tb.inv_area + p);
#pragma unroll
        for (int u = 0; u < 4; ++u) L[i * nv + k + u] = acc[u] * ia;
    }
}

bool aligned(const void *p, size_t bytes) { return ((uintptr_t)p & (bytes - 1)) == 0; }

template <typename T> const FvTables<T> &pick(const bz_mesh *m);
template <> const FvTables<double> &pick<double>(const bz_mesh *m) { return m->t64; }
template <> const FvTables<float> &pick<float>(const bz_mesh *m) { return m->t32; }
template <typename T> const T *wall_params(const bz_mesh *m);
template <> const double *wall_params<double>(const bz_mesh *m) { return m->d_wall64; }
template <> const float *wall_params<float>(const bz_mesh *m) { return m->d_wall32; }

FvIdx indices(const bz_mesh *m) {
    return FvIdx{m->d_order, m->d_meta, m->d_fid, m->d_two, m->d_ncen, m->d_cen, m->d_nsec, m->d_sec};
}


dim3 cell_grid(const bz_mesh *m, int nv, int vec) {
    return dim3((unsigned)m->n_cells, (unsigned)((nv / vec + kFvThreads - 1) / kFvThreads));
}

int fv_sm_count() {
    static std::atomic<int> cache[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64) {
        const int c = cache[dev].load(std::memory_order_relaxed);
        if (c > 0) return c;
    }
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 1;
    if (dev >= 0 && dev < 64) cache[dev].store(n, std::memory_order_relaxed);
    return n;
}

template <typename T, int VEC, int MAXF>
void faces_launch(const bz_mesh *m, const GridView &g, const T *f, T *FX, cudaStream_t st) {
    const int nv = (int)g.nv;
    const dim3 grid = cell_grid(m, nv, VEC);
    if (m->order == 3)
        fv_faces_kernel<T, VEC, MAXF, kFvCoef3, kFvCentral3><<<grid, kFvThreads, 0, st>>>(
            f, FX, pick<T>(m), indices(m), m->n_rows, nv, g.N, (T)g.L, (T)g.dv);
    else
        fv_faces_kernel<T, VEC, MAXF, 2, kFvCentral><<<grid, kFvThreads, 0, st>>>(
            f, FX, pick<T>(m), indices(m), m->n_rows, nv, g.N, (T)g.L, (T)g.dv);
}

// Threads of a block of the value passes, no more than a row needs as far as
// that goes (a row of 16^2 has 64), and their persistent grid: as many warps
// per SM as cps blocks of kFvThreads.  Transport of 19802 triangles with 256
// threads at every size and as here: 16^2 97 and 45 us, 24^2 117 and 97 us.
// The flux pass takes two thirds of them while the value rows stay in L2 (64 MB of
// 129): 24^2 on 4050 cells 26.8 and 25.7 us; on 12800, out of L2, 66.0 and 69.4.
int values_threads(int nv) { return nv <= 256 ? 64 : nv <= 512 ? 128 : nv <= 640 ? 160 : kFvThreads; }
dim3 values_grid(const bz_mesh *m, int nv, int cps) {
    const int bt = values_threads(nv), gy = (nv / 4 + bt - 1) / bt;
    int b = cps * kFvThreads / bt;
    if (cps == kFluxCtasPerSm && bt < kFvThreads && 12 * m->n_cells * nv <= (64 << 20)) b = b * 2 / 3;
    const int64_t blocks = (int64_t)fv_sm_count() * b / gy;
    return dim3((unsigned)std::max<int64_t>(1, std::min<int64_t>(m->n_cells, blocks)), (unsigned)gy);
}
template <int BT>
void values_launch(const bz_mesh *m, const GridView &g, const float *f, float *FV, cudaStream_t st) {
    const int nv = (int)g.nv;
    fv_values_persist_kernel<BT><<<values_grid(m, nv, kFacesCtasPerSm), BT, face_stage_bytes(BT), st>>>(
        f, FV, m->t32, indices(m), m->d_tripos, m->n_cells, nv);
}
// Degree 2 on FP32 triangles: a block per cell, or the staged form.  Blocks per
// cell are placed as SMs fall free and leave no lanes of a row idle beyond a block;
// the staged form hides the latency of large meshes better where a row fills one
// block.  Transport with blocks per cell and staged, us: 32^2 on 472, 2512, 7074,
// 19802 cells 17.8 and 22.0, 38.3 and 40.8, 98.7 and 96.8, 253.7 and 242.7; 24^2
// on 472, 5300, 12643, 19802 cells 15.1 and 16.5, 44.9 and 48.9, 107.7 and 106.1,
// 163.5 and 160.3; on 19802 cells 16^2 74.2 and 76.8, 20^2 127.2 and 134.3, 28^2
// 232.0 and 232.1; 36^2 on 12643 cells 228 and 293, 64^2 on 5300 cells 253 and 269.
bool faces3_staged(const bz_mesh *m, int nv) {
    const int bt = values_threads(nv);
    return m->n_cells >= (int64_t)45 * fv_sm_count() && bt >= 160 && nv <= 4 * bt && 10 * nv >= 9 * 4 * bt;
}
template <int BT, bool TWO>
void faces3_launch(const bz_mesh *m, const GridView &g, const float *f, float *FX, cudaStream_t st) {
    const int nv = (int)g.nv;
    const int64_t rows = TWO ? 0 : m->n_rows;
    if constexpr (BT >= 160) {
        if (faces3_staged(m, nv)) {
            fv_faces3_persist_kernel<BT, TWO><<<values_grid(m, nv, faces3_ctas_per_sm(BT)), BT, faces3_stage_bytes(BT), st>>>(
                f, FX, m->t32, indices(m), rows, m->n_cells, nv, g.N, (float)g.L, (float)g.dv);
            return;
        }
    }
    fv_faces3_cell_kernel<BT, TWO><<<dim3((unsigned)m->n_cells, (unsigned)((nv / 4 + BT - 1) / BT)), BT, 0, st>>>(
        f, FX, m->t32, indices(m), rows, nv, g.N, (float)g.L, (float)g.dv);
}
template <bool TWO>
void faces3_launch(const bz_mesh *m, const GridView &g, const float *f, float *FX, cudaStream_t st) {
    switch (values_threads((int)g.nv)) {
        case 64: return faces3_launch<64, TWO>(m, g, f, FX, st);
        case 128: return faces3_launch<128, TWO>(m, g, f, FX, st);
        case 160: return faces3_launch<160, TWO>(m, g, f, FX, st);
    }
    faces3_launch<kFvThreads, TWO>(m, g, f, FX, st);
}
// The flux pass starts while the reconstruction's last blocks end (on 760 to
// 19802 triangles x 32^2 it saves 2 to 3 us), except with narrow blocks on larger
// meshes: beside those of the reconstruction they would be placed unevenly.  With
// and without, us: 24^2 on 1105, 1298 cells 12.9 and 15.3, 14.5 and 16.3; 20^2 on
// 1506, 2821, 3957, 7074 cells 14.3 and 15.8, 20.6 and 20.6, 25.1 and 22.7, 38.6 and
// 33.6; 16^2 on 3957, 19802 cells 14.8 and 16.4, 50.3 and 45.3.
template <int BT>
cudaError_t flux_values_launch(const bz_mesh *m, const GridView &g, const float *FV, float *L, cudaStream_t st) {
    const int nv = (int)g.nv;
    return launch_after(fv_flux_values_persist_kernel<BT>, values_grid(m, nv, kFluxCtasPerSm), BT, face_stage_bytes(BT), st,
                        BT == kFvThreads || m->n_cells * nv <= (5 << 18), FV, L, m->t32, m->d_tripos, m->n_cells, nv, g.N, (float)g.L, (float)g.dv);
}

// FP64 takes one velocity per thread (the FP64 pipe is the bound, so loads per
// velocity cost nothing); FP32 two, and four on triangles with 4 | N, as far
// as the alignment of the caller's f allows (FX is the library's).
template <typename T>
cudaError_t faces(const bz_mesh *m, const GridView &g, const T *f, T *FX, cudaStream_t st) {
    if (m->n_cells <= 0) return cudaSuccess;
    const int nv = (int)g.nv;
    const bool tri = m->max_faces <= 3;
    if constexpr (sizeof(T) == 8) {
        if (tri) faces_launch<T, 1, 3>(m, g, f, FX, st);
        else faces_launch<T, 1, kFvMaxFaces>(m, g, f, FX, st);
    } else {
        if (tri && g.N % 4 == 0 && aligned(f, 16)) {
            if (m->order == 3)
                faces3_launch<false>(m, g, f, FX, st);
            else
                fv_faces_kernel<T, 4, 3, 2, kFvCentral><<<cell_grid(m, nv, 4), kFvThreads, 0, st>>>(
                    f, FX, m->t32, indices(m), m->n_rows, nv, g.N, (float)g.L, (float)g.dv);
        } else if (aligned(f, 8)) {
            if (tri) faces_launch<T, 2, 3>(m, g, f, FX, st);
            else faces_launch<T, 2, kFvMaxFaces>(m, g, f, FX, st);
        } else {
            if (tri) faces_launch<T, 1, 3>(m, g, f, FX, st);
            else faces_launch<T, 1, kFvMaxFaces>(m, g, f, FX, st);
        }
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && m->n_walls > 0) {
        if (!fv_walls_supported(m, g)) return cudaErrorInvalidValue;
        fv_wall_faces_kernel<T><<<(unsigned)m->n_walls, kFvThreads, 0, st>>>(
            FX, pick<T>(m), m->d_fid, m->d_wall, m->d_wallslot, wall_params<T>(m), nv, g.N, (T)g.L, (T)g.dv);
        e = cudaGetLastError();
    }
    return e;
}

template <typename T, int VEC, int MAXF>
cudaError_t sum_launch(const bz_mesh *m, const GridView &g, const T *FX, T *L, cudaStream_t st) {
    const int nv = (int)g.nv;
    const dim3 grid = cell_grid(m, nv, VEC);
    const int *wall = m->n_walls > 0 ? m->d_wall : nullptr;
    if (m->order == 3)
        return launch_after(fv_sum_kernel<T, VEC, MAXF, kFvCoef3>, grid, kFvThreads, 0, st, true, FX, L, pick<T>(m),
                            indices(m), wall, m->n_rows, nv, g.N, 1.f / (float)g.N, (T)g.L, (T)g.dv);
    return launch_after(fv_sum_kernel<T, VEC, MAXF, 2>, grid, kFvThreads, 0, st, true, FX, L, pick<T>(m), indices(m),
                        wall, m->n_rows, nv, g.N, 1.f / (float)g.N, (T)g.L, (T)g.dv);
}

// 16-byte rows where L allows (N^2 is a multiple of 4)
template <typename T>
cudaError_t sum(const bz_mesh *m, const GridView &g, const T *FX, T *L, cudaStream_t st) {
    if (m->n_cells <= 0) return cudaSuccess;
    constexpr int V = 16 / (int)sizeof(T);
    const bool tri = m->max_faces <= 3, al = aligned(L, 16);
    return tri && al ? sum_launch<T, V, 3>(m, g, FX, L, st)
           : tri     ? sum_launch<T, 1, 3>(m, g, FX, L, st)
           : al      ? sum_launch<T, V, kFvMaxFaces>(m, g, FX, L, st)
                     : sum_launch<T, 1, kFvMaxFaces>(m, g, FX, L, st);
}

template <typename T, int VEC, int MAXF>
void first_launch(const bz_mesh *m, const GridView &g, const T *f, T *L, cudaStream_t st) {
    fv_first_kernel<T, VEC, MAXF><<<cell_grid(m, (int)g.nv, VEC), kFvThreads, 0, st>>>(
        f, L, pick<T>(m), indices(m), m->d_nb, (int)g.nv, g.N, (T)g.L, (T)g.dv);
}

template <typename T>
cudaError_t first(const bz_mesh *m, const GridView &g, const T *f, T *L, cudaStream_t st) {
    if (m->n_cells <= 0) return cudaSuccess;
    const bool tri = m->max_faces <= 3;
    if (m->n_walls > 0) {
        if (!fv_walls_supported(m, g)) return cudaErrorInvalidValue;
        const unsigned grid = (unsigned)m->n_cells;
        if (tri)
            fv_first_wall_kernel<T, 3><<<grid, kFvThreads, 0, st>>>(f, L, pick<T>(m), indices(m), m->d_nb, m->d_wall,
                                                                    wall_params<T>(m), (int)g.nv, g.N, (T)g.L, (T)g.dv);
        else
            fv_first_wall_kernel<T, kFvMaxFaces><<<grid, kFvThreads, 0, st>>>(
                f, L, pick<T>(m), indices(m), m->d_nb, m->d_wall, wall_params<T>(m), (int)g.nv, g.N, (T)g.L, (T)g.dv);
        return cudaGetLastError();
    }
    if (tri && g.N % 4 == 0 && aligned(f, 16) && aligned(L, 16)) first_launch<T, 4, 3>(m, g, f, L, st);
    else if (tri) first_launch<T, 1, 3>(m, g, f, L, st);
    else first_launch<T, 1, kFvMaxFaces>(m, g, f, L, st);
    return cudaGetLastError();
}

}  // namespace

// The two-sided passes (see fv_two_sided): FX rows [face][side][point].
cudaError_t launch_fv_faces_two_f32(const bz_mesh *m, const GridView &g, const float *f, float *FX, cudaStream_t st) {
    if (m->n_cells <= 0) return cudaSuccess;
    const int nv = (int)g.nv;
    auto launch = [&](auto kernel, int vec) {
        kernel<<<cell_grid(m, nv, vec), kFvThreads, 0, st>>>(f, FX, m->t32, indices(m), 0, nv, g.N, (float)g.L, (float)g.dv);
    };
    const bool tri = m->max_faces <= 3;
    if (tri && g.N % 4 == 0 && aligned(f, 16)) faces3_launch<true>(m, g, f, FX, st);
    else if (tri) launch(fv_faces_kernel<float, 1, 3, kFvCoef3, kFvCentral3, true>, 1);
    else if (aligned(f, 8)) launch(fv_faces_kernel<float, 2, kFvMaxFaces, kFvCoef3, kFvCentral3, true>, 2);
    else launch(fv_faces_kernel<float, 1, kFvMaxFaces, kFvCoef3, kFvCentral3, true>, 1);
    return cudaGetLastError();
}
cudaError_t launch_fv_sum_two_f32(const bz_mesh *m, const GridView &g, const float *FX, float *L, cudaStream_t st) {
    if (m->n_cells <= 0) return cudaSuccess;
    const int nv = (int)g.nv;
    auto launch = [&](auto kernel, int vec) {
        return launch_after(kernel, cell_grid(m, nv, vec), kFvThreads, 0, st, true, FX, L, m->t32, indices(m), nv, g.N,
                            (float)g.L, (float)g.dv);
    };
    if (g.N % 4 || !aligned(L, 16)) return launch(fv_sum_two_kernel<1, kFvMaxFaces>, 1);
    return m->max_faces <= 3 ? launch(fv_sum_two_kernel<4, 3>, 4) : launch(fv_sum_two_kernel<4, kFvMaxFaces>, 4);
}

cudaError_t fv_values_setup() {
    const std::pair<const void *, size_t> big[] = {
        {(const void *)fv_values_persist_kernel<kFvThreads>, face_stage_bytes(kFvThreads)},
        {(const void *)fv_flux_values_persist_kernel<kFvThreads>, face_stage_bytes(kFvThreads)},
        {(const void *)fv_faces3_persist_kernel<kFvThreads, false>, faces3_stage_bytes(kFvThreads)},
        {(const void *)fv_faces3_persist_kernel<kFvThreads, true>, faces3_stage_bytes(kFvThreads)}};
    cudaError_t e = cudaSuccess;
    for (const auto &[kernel, bytes] : big)
        if (e == cudaSuccess) e = allow_dynamic_smem(kernel, bytes);
    return e;
}

bool fv_value_mode(const bz_mesh *m, const GridView &g, const void *f, const void *L) {
    return m->d_tripos && m->n_walls == 0 && g.N % 4 == 0 && aligned(f, 16) && aligned(L, 16);
}

bool fv_two_sided(const bz_mesh *m, bool f32) { return f32 && m->order == 3 && m->n_two > 0 && m->n_walls == 0; }

int64_t fv_scratch_rows(const bz_mesh *m, bool f32, bool step) {
    if (m->order == 1) return 0;
    if (step && fv_two_sided(m, f32)) return 4 * m->n_rows;
    const int64_t flux = m->n_rows + (f32 ? m->n_two * (m->order == 3 ? 4 : 2) : 0);
    return f32 && m->d_tripos ? std::max<int64_t>(flux, 3 * m->n_cells) : flux;
}

cudaError_t launch_fv_values_f32(const bz_mesh *m, const GridView &g, const float *f, float *FV, cudaStream_t st) {
    if (m->n_cells <= 0) return cudaSuccess;
    switch (values_threads((int)g.nv)) {
        case 64: values_launch<64>(m, g, f, FV, st); break;
        case 128: values_launch<128>(m, g, f, FV, st); break;
        case 160: values_launch<160>(m, g, f, FV, st); break;
        default: values_launch<kFvThreads>(m, g, f, FV, st);
    }
    return cudaGetLastError();
}
cudaError_t launch_fv_flux_values_f32(const bz_mesh *m, const GridView &g, const float *FV, float *L,
                                      cudaStream_t st) {
    if (m->n_cells <= 0) return cudaSuccess;
    switch (values_threads((int)g.nv)) {
        case 64: return flux_values_launch<64>(m, g, FV, L, st);
        case 128: return flux_values_launch<128>(m, g, FV, L, st);
        case 160: return flux_values_launch<160>(m, g, FV, L, st);
        default: return flux_values_launch<kFvThreads>(m, g, FV, L, st);
    }
}

bool fv_walls_supported(const bz_mesh *m, const GridView &g) {
    return m->n_walls == 0 || (g.N % 4 == 0 && g.nv <= 4 * kFvThreads);
}

cudaError_t launch_fv_first_f64(const bz_mesh *m, const GridView &g, const double *f, double *L, cudaStream_t st) {
    return first<double>(m, g, f, L, st);
}
cudaError_t launch_fv_first_f32(const bz_mesh *m, const GridView &g, const float *f, float *L, cudaStream_t st) {
    return first<float>(m, g, f, L, st);
}
cudaError_t launch_fv_faces_f64(const bz_mesh *m, const GridView &g, const double *f, double *FX, cudaStream_t st) {
    return faces<double>(m, g, f, FX, st);
}
cudaError_t launch_fv_faces_f32(const bz_mesh *m, const GridView &g, const float *f, float *FX, cudaStream_t st) {
    return faces<float>(m, g, f, FX, st);
}
cudaError_t launch_fv_sum_f64(const bz_mesh *m, const GridView &g, const double *FX, double *L, cudaStream_t st) {
    return sum<double>(m, g, FX, L, st);
}
cudaError_t launch_fv_sum_f32(const bz_mesh *m, const GridView &g, const float *FX, float *L, cudaStream_t st) {
    return sum<float>(m, g, FX, L, st);
}

}  // namespace bz
