// FP32 mode products on the CUDA cores; FP64 kernels: the stencil form of the
// Kronecker-sum action with the reaction term, the pointwise stage kernels of EXPRK3DS_REAL and the phi-function evaluation.
#include <math.h>

#include <algorithm>
#include <vector>

#include "mm64.h"

namespace ds {

// ---------------------------------------------------------------------------
// FP32 mode products on the CUDA cores: Y(i, f) = sum over terms of alpha sum_j
// L(i, j) X(j, f) (+ Y) over the fibres f of a mode, entry (j, f) of a tensor at
// (f / I) (I n) + f % I + I j.  A block takes up to 128 rows i (a multiple of
// eight, n cut evenly, so that n = 100 pads to 104) by 64 fibres, counted through
// all slices; a thread 8 x 8 outputs, 64 FMAs per four 16-byte shared-memory
// loads, each output one FMA chain in ascending j.  The next 16 entries of the
// contraction are fetched while the current ones are used.  One product of 10^6
// points is 16k threads, a third of what the SMs hold at 8 x 8 outputs each, so
// the products of a phase share a launch (FitzHugh-Nagumo 100^3, two steps: 3.25 ms
// with 64 x 64 tiles of 4 x 4 outputs per thread and a launch per product, 5.8 with
// this tile and a launch per product, 2.14 so; tried and left out, 4 x 8 outputs per
// thread where a launch has two products: 2.24).  18 products of 100 entries each run at 21 TFLOP/s, the FMA pipe
// 43 % busy: the padding (104 of 100 rows, 112 of 100 entries) and the copies'
// addresses take the rest.
// ---------------------------------------------------------------------------
namespace {
constexpr int kSgRows = 128, kSgCols = 64, kSgK = 16, TR = 8;   // TR: rows per thread

struct SProd {
    int n, rows;          // contracted size; rows per block
    int64_t I, fibres;
    int64_t sLi, sLj;
    bool wide_l, wide_x;  // rows of L, fibres of X in aligned groups of four
    F32Product p[kMaxProducts32];
};

__global__ void __launch_bounds__(kSgRows, 4) k_mode_f32(const __grid_constant__ SProd g)
{
    __shared__ __align__(16) float Ls[2][kSgK][kSgRows + 4];
    __shared__ __align__(16) float Xs[2][kSgK][kSgCols + 4];
    __shared__ int64_t off[kSgCols];
    const F32Product &p = g.p[blockIdx.z];
    const int t = threadIdx.x, nt = blockDim.x, rows = g.rows;
    const int64_t f0 = (int64_t)blockIdx.x * kSgCols;
    const int i0 = blockIdx.y * rows;
    for (int c = t; c < kSgCols; c += nt) {
        const int64_t f = f0 + c, o = f / g.I;
        off[c] = f < g.fibres ? o * (g.I * g.n) + (f - o * g.I) : -1;
    }
    __syncthreads();
    const int tx = t % 8, ti = t / 8;   // fibres 4 tx .. and 32 + 4 tx .., rows TR ti ..
    const bool li_fast = g.sLi == 1, x_fast = g.I > 1;
    // The next chunk's copies run behind the FMAs; out-of-range entries arrive as
    // zero.  Four entries per copy where rows (fibres) of four are aligned; else
    // single ones, eight lanes along the fast index.
    auto copy4 = [](float *dst, const float *src, bool ok) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                     "l"(src), "r"(ok ? 4 : 0)
                     : "memory");
    };
    auto copy16 = [](float *dst, const float *src, bool ok) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                     "l"(src), "r"(ok ? 16 : 0)
                     : "memory");
    };
    const int step = nt / 8, quads = rows / 4;
    auto fill = [&](int buf, const float *X, const float *L, int k0) {
        if (g.wide_l) {
            for (int k = t / quads, i = t % quads * 4; k < kSgK;) {
                const bool in = k0 + k < g.n && i0 + i < g.n;
                copy16(&Ls[buf][k][i], in ? L + i0 + i + (int64_t)(k0 + k) * g.n : L, in);
                i += 4 * nt;   // the next of this thread's quads
                while (i >= rows) i -= rows, ++k;
            }
        } else if (li_fast) {
            for (int i = t; i < rows; i += nt)
#pragma unroll
                for (int k = 0; k < kSgK; ++k) {
                    const bool in = i0 + i < g.n && k0 + k < g.n;
                    copy4(&Ls[buf][k][i], in ? L + i0 + i + (k0 + k) * g.sLj : L, in);
                }
        } else {
            for (int i = ti; i < rows; i += step)
#pragma unroll
                for (int k = tx; k < kSgK; k += 8) {
                    const bool in = k0 + k < g.n && i0 + i < g.n;
                    copy4(&Ls[buf][k][i], in ? L + (i0 + i) * g.sLi + (k0 + k) * g.sLj : L, in);
                }
        }
        if (g.wide_x) {
            for (int e = t; e < kSgK * kSgCols / 4; e += nt) {
                const int k = e / (kSgCols / 4), c = e % (kSgCols / 4) * 4;
                const int64_t o = off[c];
                const bool in = k0 + k < g.n && o >= 0;
                copy16(&Xs[buf][k][c], in ? X + o + g.I * (k0 + k) : X, in);
            }
        } else if (x_fast) {
            for (int k = ti; k < kSgK; k += step)
#pragma unroll
                for (int c = tx; c < kSgCols; c += 8) {
                    const int64_t o = off[c];
                    const bool in = k0 + k < g.n && o >= 0;
                    copy4(&Xs[buf][k][c], in ? X + o + g.I * (k0 + k) : X, in);
                }
        } else {
            for (int c = ti; c < kSgCols; c += step) {
                const int64_t o = off[c];
#pragma unroll
                for (int k = tx; k < kSgK; k += 8) {
                    const bool in = k0 + k < g.n && o >= 0;
                    copy4(&Xs[buf][k][c], in ? X + o + k0 + k : X, in);
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto landed = [] {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
    };
    for (int term = 0; term < p.nterm; ++term) {
        const float *X = p.X[term], *L = p.L[term], alpha = p.alpha[term];
        float acc[TR][8];
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[r][c] = 0.0f;
        fill(0, X, L, 0);
        landed();
        int buf = 0;
        for (int k0 = 0; k0 < g.n; k0 += kSgK) {
            if (k0 + kSgK < g.n) fill(buf ^ 1, X, L, k0 + kSgK);
#pragma unroll 4
            for (int k = 0; k < kSgK; ++k) {
                float a[TR];
#pragma unroll
                for (int r = 0; r < TR; r += 4)
                    *reinterpret_cast<float4 *>(&a[r]) = *reinterpret_cast<const float4 *>(&Ls[buf][k][ti * TR + r]);
                const float4 b0 = *reinterpret_cast<const float4 *>(&Xs[buf][k][tx * 4]);
                const float4 b1 = *reinterpret_cast<const float4 *>(&Xs[buf][k][32 + tx * 4]);
                const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
                for (int r = 0; r < TR; ++r)
#pragma unroll
                    for (int c = 0; c < 8; ++c) acc[r][c] = fmaf(a[r], b[c], acc[r][c]);
            }
            landed();
            buf ^= 1;
        }
        // a thread adds its own outputs' terms, in order
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int64_t o = off[(c < 4 ? 0 : 28) + tx * 4 + c];
            if (o < 0) continue;
#pragma unroll
            for (int r = 0; r < TR; ++r) {
                const int i = i0 + ti * TR + r;
                if (ti * TR + r >= rows || i >= g.n) continue;
                float *y = p.Y + o + g.I * i;
                *y = term > 0 || p.accumulate ? __fmaf_rn(alpha, acc[r][c], *y) : __fmul_rn(alpha, acc[r][c]);
            }
        }
    }
}
}  // namespace

int launch_products_f32(int d, const int64_t *n, int mu, int transpose, const F32Product *p, int count, cudaStream_t st)
{
    SProd g{};
    g.n = (int)n[mu];
    g.I = g.fibres = 1;
    for (int q = 0; q < d; ++q) {
        if (q < mu) g.I *= n[q];
        if (q != mu) g.fibres *= n[q];
    }
    g.sLi = transpose ? n[mu] : 1;
    g.sLj = transpose ? 1 : n[mu];
    g.wide_l = !transpose && g.n % 4 == 0;
    g.wide_x = g.I % 4 == 0;
    for (int q = 0; q < count; ++q)
        for (int t = 0; t < p[q].nterm; ++t) {
            g.wide_l = g.wide_l && ((uintptr_t)p[q].L[t] & 15) == 0;
            g.wide_x = g.wide_x && ((uintptr_t)p[q].X[t] & 15) == 0;
        }
    const int blocks = (g.n + kSgRows - 1) / kSgRows;
    g.rows = ((g.n + blocks - 1) / blocks + 7) / 8 * 8;
    int launches = 0;
    for (int q = 0; q < count; q += kMaxProducts32, ++launches) {
        const int m = std::min(kMaxProducts32, count - q);
        std::copy(p + q, p + q + m, g.p);
        const dim3 grid((unsigned)((g.fibres + kSgCols - 1) / kSgCols), (unsigned)((g.n + g.rows - 1) / g.rows), m);
        k_mode_f32<<<grid, std::max(32, g.rows), 0, st>>>(g);
    }
    return launches;
}

// ---------------------------------------------------------------------------
// Reaction terms (Section 3 models).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void react(const Model &m, double u, double v, double &gu, double &gv)
{
    if (m.model == DS_SCHNAKENBERG) {
        const double u2v = u * u * v;
        gu = m.p[0] * ((m.p[1] - u) + u2v);
        gv = m.p[0] * (m.p[2] - u2v);
    } else if (m.model == DS_FHN) {
        gu = fma(-u * u, u, u - v);
        gv = m.p[0] * fma(-m.p[1], v, u - m.p[2]);
    } else {
        gu = 0.0;
        gv = 0.0;
    }
}

// g(u + du, v + dv) - g(u, v) as the polynomial in the increments: no
// cancellation, and fewer operations than g twice (the pointwise kernels are
// bound by the FP64 pipe, 16 clocks per warp instruction and SM)
__device__ __forceinline__ void react_difference(const Model &m, double u, double v, double du, double dv, double &Du,
                                                 double &Dv)
{
    if (m.model == DS_SCHNAKENBERG) {
        const double q = du * fma(2.0, u, du);                  // (u + du)^2 - u^2
        const double w = fma(q, v + dv, u * u * dv);            // (u + du)^2 (v + dv) - u^2 v
        Du = m.p[0] * (w - du);
        Dv = -m.p[0] * w;
    } else if (m.model == DS_FHN) {
        const double c = fma(3.0 * u, u + du, du * du);         // ((u + du)^3 - u^3) / du
        Du = fma(-du, c, du - dv);
        Dv = m.p[0] * fma(-m.p[1], dv, du);
    } else {
        Du = 0.0;
        Dv = 0.0;
    }
}

namespace {
// K U for one point of one component: each tridiagonal row as lo (u- - u) + up (u+ -
// u) + (row sum) u, so that a constant state gives exactly zero where the rows sum
// to zero, and neighbouring values lose nothing in their difference; all in one
// chain of FMAs.  Where the outer bands outweigh the diagonal (advection) the
// differences would bring in |lo| |u|, which the row itself does not have: such a
// direction takes lo u- + up u+ + di u (plain; `sum` is its diagonal).  IT: 32-bit
// indices where the grid allows them.
template <typename IT>
__device__ __forceinline__ double stencil_point(const Stencil &s, const double *U, IT p)
{
    const double u = U[p];
    double acc = 0.0;
    IT stride = 1, rest = p;
#pragma unroll
    for (int mu = 0; mu < kMaxD; ++mu) {
        if (mu < s.d) {
            const IT nm = (IT)s.n[mu], q = rest / nm, i = rest - q * nm;
            rest = q;
            const double from = s.plain[mu] ? 0.0 : u;
            if (i > 0) acc = fma(s.lo[mu][i], U[p - stride] - from, acc);
            if (i + 1 < nm) acc = fma(s.up[mu][i], U[p + stride] - from, acc);
            const double rs = s.sum[mu][i];
            if (__double_as_longlong(rs)) acc = fma(rs, u, acc);
            stride *= nm;
        }
    }
    return acc;
}

template <typename IT>
__global__ void k_kronsum_f64(Stencil s, IT N, const double *__restrict__ X, double *__restrict__ Y)
{
    pdl_trigger();
    pdl_wait();
    for (IT p = (IT)blockIdx.x * blockDim.x + threadIdx.x; p < N; p += (IT)gridDim.x * blockDim.x)
        Y[p] = stencil_point<IT>(s, X, p);
}

template <typename IT>
__global__ void k_rhs_f64(Stencil s0, Stencil s1, Model m, IT N, const double *__restrict__ U,
                          double *__restrict__ F)
{
    pdl_trigger();
    pdl_wait();
    for (IT p = (IT)blockIdx.x * blockDim.x + threadIdx.x; p < N; p += (IT)gridDim.x * blockDim.x) {
        double gu, gv;
        react(m, U[p], U[N + p], gu, gv);
        F[p] = stencil_point<IT>(s0, U, p) + gu;
        F[N + p] = stencil_point<IT>(s1, U + N, p) + gv;
    }
}

__global__ void k_stage_diff_f64(Model m, int64_t N, const double *__restrict__ U,
                                 const double *__restrict__ a, double w1,
                                 const double *__restrict__ b, double w2, double *__restrict__ D)
{
    pdl_trigger();
    pdl_wait();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < N;
         p += (int64_t)gridDim.x * blockDim.x) {
        double du = w1 * a[p], dv = w1 * a[N + p];
        if (b) {
            du = fma(w2, b[p], du);
            dv = fma(w2, b[N + p], dv);
        }
        react_difference(m, U[p], U[N + p], du, dv, D[p], D[N + p]);
    }
}

__global__ void k_final_f64(int64_t n2, double *__restrict__ U, const double *__restrict__ a,
                            double w1, const double *__restrict__ b, double w2)
{
    pdl_trigger();
    pdl_wait();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n2;
         p += (int64_t)gridDim.x * blockDim.x)
        U[p] = fma(w2, b[p], fma(w1, a[p], U[p]));
}

__global__ void k_add_g_f64(Model m, int64_t N, const double *__restrict__ U, double *__restrict__ F)
{
    pdl_trigger();
    pdl_wait();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < N;
         p += (int64_t)gridDim.x * blockDim.x) {
        double gu, gv;
        react(m, U[p], U[N + p], gu, gv);
        F[p] = __dadd_rn(F[p], gu);
        F[N + p] = __dadd_rn(F[N + p], gv);
    }
}

__global__ void k_nonfinite(const double *x, int64_t count, int *flag)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < count;
         p += (int64_t)gridDim.x * blockDim.x)
        if (!isfinite(x[p])) atomicExch(flag, 1);
}

// J_g(U)^T lam for one point; model as in react()
__device__ __forceinline__ void jacT(const Model &m, double u, double v, double lu, double lv, double &ou,
                                     double &ov)
{
    double juu, juv, jvu, jvv;
    if (m.model == DS_SCHNAKENBERG) {
        juu = m.p[0] * (-1.0 + 2.0 * u * v);
        juv = m.p[0] * u * u;
        jvu = -2.0 * m.p[0] * u * v;
        jvv = -m.p[0] * u * u;
    } else if (m.model == DS_FHN) {
        juu = 1.0 - 3.0 * u * u;
        juv = -1.0;
        jvu = m.p[0];
        jvv = -m.p[0] * m.p[1];
    } else {
        juu = juv = jvu = jvv = 0.0;
    }
    ou = juu * lu + jvu * lv;
    ov = juv * lu + jvv * lv;
}

// (dg/dp)(U)^T lam for one point: contributions to the three model parameters
__device__ __forceinline__ void dparam_point(const Model &m, double u, double v, double lu, double lv,
                                             double &d0, double &d1, double &d2)
{
    if (m.model == DS_SCHNAKENBERG) {
        d0 = (m.p[1] - u + u * u * v) * lu + (m.p[2] - u * u * v) * lv;
        d1 = m.p[0] * lu;
        d2 = m.p[0] * lv;
    } else if (m.model == DS_FHN) {
        d0 = (u - m.p[1] * v - m.p[2]) * lv;
        d1 = -m.p[0] * v * lv;
        d2 = -m.p[0] * lv;
    } else {
        d0 = d1 = d2 = 0.0;
    }
}

// Y = U + w1 a (+ w2 b), 2 N values
// (Y may be U)
__global__ void k_axpy2(int64_t n2, const double *U, const double *__restrict__ a, double w1,
                        const double *__restrict__ b, double w2, double *Y)
{
    pdl_trigger();
    pdl_wait();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n2;
         p += (int64_t)gridDim.x * blockDim.x) {
        double y = fma(w1, a[p], U[p]);
        if (b) y = fma(w2, b[p], y);
        Y[p] = y;
    }
}

// D = g(Us) - g(U)
__global__ void k_gdiff(Model m, int64_t N, const double *__restrict__ U, const double *__restrict__ Us,
                        double *__restrict__ D)
{
    pdl_trigger();
    pdl_wait();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < N;
         p += (int64_t)gridDim.x * blockDim.x) {
        const double u = U[p], v = U[N + p];
        react_difference(m, u, v, Us[p] - u, Us[N + p] - v, D[p], D[N + p]);
    }
}

// out = J_g(Us)^T lam
__global__ void k_jacT(Model m, int64_t N, const double *__restrict__ Us, const double *__restrict__ lam,
                       double *__restrict__ out)
{
    pdl_trigger();
    pdl_wait();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < N;
         p += (int64_t)gridDim.x * blockDim.x) {
        double ou, ov;
        jacT(m, Us[p], Us[N + p], lam[p], lam[N + p], ou, ov);
        out[p] = ou;
        out[N + p] = ov;
    }
}

// K^T x for one point of one component (transposed tridiagonal rows)
template <typename IT>
__device__ __forceinline__ double stencil_point_T(const Stencil &s, const double *X, IT p)
{
    double acc = 0.0;
    IT stride = 1, rest = p;
#pragma unroll
    for (int mu = 0; mu < kMaxD; ++mu) {
        if (mu < s.d) {
            const IT nm = (IT)s.n[mu], q = rest / nm, i = rest - q * nm;
            rest = q;
            acc = fma(s.di[mu][i], X[p], acc);
            if (i > 0) acc = fma(s.up[mu][i - 1], X[p - stride], acc);
            if (i + 1 < nm) acc = fma(s.lo[mu][i + 1], X[p + stride], acc);
            stride *= nm;
        }
    }
    return acc;
}

template <typename IT>
__global__ void k_kronsumT(Stencil s0, Stencil s1, IT N, const double *__restrict__ X, double *__restrict__ Y)
{
    pdl_trigger();
    pdl_wait();
    for (IT p = (IT)blockIdx.x * blockDim.x + threadIdx.x; p < N; p += (IT)gridDim.x * blockDim.x) {
        Y[p] = stencil_point_T<IT>(s0, X, p);
        Y[N + p] = stencil_point_T<IT>(s1, X + N, p);
    }
}

// lam_n = lam + lU3 + lU2 + KT + J_g(U)^T (lF - lD2 - lD3); dp += the three
// parameter gradients (block reduction, one atomic per block and parameter)
__global__ void __launch_bounds__(256) k_adjoint_final(Model m, int64_t N, const double *__restrict__ U,
                                                       const double *__restrict__ U2,
                                                       const double *__restrict__ U3,
                                                       const double *__restrict__ lam,
                                                       const double *__restrict__ lU3,
                                                       const double *__restrict__ lU2,
                                                       const double *__restrict__ KT,
                                                       const double *__restrict__ lF,
                                                       const double *__restrict__ lD2,
                                                       const double *__restrict__ lD3,
                                                       double *__restrict__ lam_n, double *dp)
{
    pdl_trigger();
    pdl_wait();
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < N;
         p += (int64_t)gridDim.x * blockDim.x) {
        const double gu = lF[p] - lD2[p] - lD3[p], gv = lF[N + p] - lD2[N + p] - lD3[N + p];
        double ou, ov;
        jacT(m, U[p], U[N + p], gu, gv, ou, ov);
        lam_n[p] = lam[p] + lU3[p] + lU2[p] + KT[p] + ou;
        lam_n[N + p] = lam[N + p] + lU3[N + p] + lU2[N + p] + KT[N + p] + ov;
        if (dp) {
            double a0, a1, a2;
            dparam_point(m, U[p], U[N + p], gu, gv, a0, a1, a2);
            s0 += a0; s1 += a1; s2 += a2;
            dparam_point(m, U2[p], U2[N + p], lD2[p], lD2[N + p], a0, a1, a2);
            s0 += a0; s1 += a1; s2 += a2;
            dparam_point(m, U3[p], U3[N + p], lD3[p], lD3[N + p], a0, a1, a2);
            s0 += a0; s1 += a1; s2 += a2;
        }
    }
    if (!dp) return;
    __shared__ double red[3][256];
    red[0][threadIdx.x] = s0;
    red[1][threadIdx.x] = s1;
    red[2][threadIdx.x] = s2;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int q = 0; q < 3; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int q = 0; q < 3; ++q) atomicAdd(dp + q, red[q][0]);
}

__global__ void __launch_bounds__(256) k_dot_accum(int64_t n, const double *__restrict__ a,
                                                   const double *__restrict__ b, double w, double *out)
{
    pdl_trigger();
    pdl_wait();
    double s = 0.0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x)
        s += a[p] * b[p];
    __shared__ double red[256];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(out, w * red[0]);
}

__global__ void __launch_bounds__(256) k_dot_kterm(Model m, int64_t N, const double *__restrict__ U,
                                                   const double *__restrict__ F,
                                                   const double *__restrict__ lF, double *out)
{
    pdl_trigger();
    pdl_wait();
    double s0 = 0.0, s1 = 0.0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < N;
         p += (int64_t)gridDim.x * blockDim.x) {
        double gu, gv;
        react(m, U[p], U[N + p], gu, gv);
        s0 += lF[p] * (F[p] - gu);
        s1 += lF[N + p] * (F[N + p] - gv);
    }
    __shared__ double red[2][256];
    red[0][threadIdx.x] = s0;
    red[1][threadIdx.x] = s1;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) {
            red[0][threadIdx.x] += red[0][threadIdx.x + k];
            red[1][threadIdx.x] += red[1][threadIdx.x + k];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        atomicAdd(out, red[0][0]);
        atomicAdd(out + 1, red[1][0]);
    }
}

// Threads of a block for n points: small grids take small blocks, so that every
// SM's FP64 pipe (16 clocks per warp instruction) has a share.
int block_for(int64_t n)
{
    int b = 256;
    while (b > 32 && n < 2 * 152 * (int64_t)b) b /= 2;
    return b;
}
int grid_for(int64_t n, int block = 256)
{
    int64_t b = (n + block - 1) / block;
    return (int)std::min<int64_t>(b, 152 * 16 * (256 / block));
}
}  // namespace

int launch_rhs_f64(const Stencil *s2, const Model &m, int64_t N, const double *U, double *F,
                   cudaStream_t st)
{
    const dim3 grid(grid_for(N, block_for(N))), block(block_for(N));
    // (headroom for the stride past the end)
    if (N < (int64_t)1 << 30) pdl_launch(k_rhs_f64<int>, grid, block, 0, st, s2[0], s2[1], m, (int)N, U, F);
    else pdl_launch(k_rhs_f64<int64_t>, grid, block, 0, st, s2[0], s2[1], m, N, U, F);
    return 1;
}

void launch_kronsum_f64(const Stencil &s, int64_t N, const double *X, double *Y, cudaStream_t st)
{
    pdl_launch(k_kronsum_f64<int64_t>, dim3(grid_for(N, block_for(N))), dim3(block_for(N)), 0, st, s, N, X, Y);
}

void launch_stage_diff_f64(const Model &m, int64_t N, const double *U, const double *a, double w1,
                           const double *b, double w2, double *D, cudaStream_t st)
{
    pdl_launch(k_stage_diff_f64, dim3(grid_for(N, block_for(N))), dim3(block_for(N)), 0, st, m, N, U, a, w1, b, w2, D);
}

void launch_final_f64(int64_t N, double *U, const double *a, double w1, const double *b,
                      double w2, cudaStream_t st)
{
    pdl_launch(k_final_f64, dim3(grid_for(2 * N, block_for(2 * N))), dim3(block_for(2 * N)), 0, st, 2 * N, U, a, w1, b, w2);
}

void launch_add_g_f64(const Model &m, int64_t N, const double *U, double *F, cudaStream_t st)
{
    pdl_launch(k_add_g_f64, dim3(grid_for(N, block_for(N))), dim3(block_for(N)), 0, st, m, N, U, F);
}

void launch_axpy2_f64(int64_t N, const double *U, const double *a, double w1, const double *b, double w2,
                      double *Y, cudaStream_t st)
{
    pdl_launch(k_axpy2, dim3(grid_for(2 * N, block_for(2 * N))), dim3(block_for(2 * N)), 0, st, 2 * N, U, a, w1, b, w2, Y);
}
void launch_gdiff_f64(const Model &m, int64_t N, const double *U, const double *Us, double *D, cudaStream_t st)
{
    pdl_launch(k_gdiff, dim3(grid_for(N, block_for(N))), dim3(block_for(N)), 0, st, m, N, U, Us, D);
}
void launch_jacT_f64(const Model &m, int64_t N, const double *Us, const double *lam, double *out,
                     cudaStream_t st)
{
    pdl_launch(k_jacT, dim3(grid_for(N, block_for(N))), dim3(block_for(N)), 0, st, m, N, Us, lam, out);
}
void launch_kronsumT_f64(const Stencil *s2, int64_t N, const double *X, double *Y, cudaStream_t st)
{
    const dim3 grid(grid_for(N, block_for(N))), block(block_for(N));
    if (N < (int64_t)1 << 30) pdl_launch(k_kronsumT<int>, grid, block, 0, st, s2[0], s2[1], (int)N, X, Y);
    else pdl_launch(k_kronsumT<int64_t>, grid, block, 0, st, s2[0], s2[1], N, X, Y);
}
void launch_adjoint_final_f64(const Model &m, int64_t N, const double *U, const double *U2,
                              const double *U3, const double *lam, const double *lU3, const double *lU2,
                              const double *KT, const double *lF, const double *lD2, const double *lD3,
                              double *lam_n, double *dp, cudaStream_t st)
{
    pdl_launch(k_adjoint_final, dim3(grid_for(N)), dim3(256), 0, st, m, N, U, U2, U3, lam, lU3, lU2, KT, lF, lD2, lD3, lam_n, dp);
}

void launch_dot_accum_f64(int64_t n, const double *a, const double *b, double w, double *out,
                          cudaStream_t st)
{
    pdl_launch(k_dot_accum, dim3(grid_for(n)), dim3(256), 0, st, n, a, b, w, out);
}
void launch_dot_kterm_f64(const Model &m, int64_t N, const double *U, const double *F, const double *lF,
                          double *out, cudaStream_t st)
{
    pdl_launch(k_dot_kterm, dim3(grid_for(N)), dim3(256), 0, st, m, N, U, F, lF, out);
}

void launch_nonfinite_scan(const double *x, int64_t count, int *flag, cudaStream_t st)
{
    k_nonfinite<<<grid_for(count), 256, 0, st>>>(x, count, flag);
}

// ---------------------------------------------------------------------------
// phi_0..phi_2 of a batch of n x n matrices z_b A_b by scaling, degree-16
// Taylor and the modified squaring of Skaflestad & Wright:
//   phi_0(2Y) = phi_0(Y)^2,
//   phi_1(2Y) = (phi_0(Y) phi_1(Y) + phi_1(Y)) / 2,
//   phi_2(2Y) = (phi_0(Y) phi_2(Y) + phi_1(Y) + phi_2(Y)) / 4.
// Matrix b is squared exactly s_b times, s_b the least s >= 0 with
// ||2^-s z_b A_b||_1 <= 1/2; the batch is sorted by s_b, so that each squaring
// runs on the matrices that still need it.  The Taylor polynomials in Y = 2^-s z A
// are evaluated in blocks of four powers (Paterson & Stockmeyer 1973): Y^2, then
// Y^3 and Y^4, then three Horner steps in Y^4 on the three polynomials together,
// 12 matrix products instead of one per degree.
// ---------------------------------------------------------------------------
namespace {

__global__ void k_build_X(int64_t nn, const double *const *Asrc, const double *z, double *X, int64_t stride)
{
    const int b = blockIdx.y;
    const double *A = Asrc[b];
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nn;
         e += (int64_t)gridDim.x * blockDim.x)
        X[b * stride + e] = z[b] * A[e];
}

// one block per matrix: column abs-sum maximum
__global__ void k_norm1(int n, const double *X, int64_t stride, double *out)
{
    const int b = blockIdx.x;
    const double *M = X + b * stride;
    __shared__ double red[256];
    double best = 0.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        double s = 0.0;
        for (int i = 0; i < n; ++i) s += fabs(M[i + (int64_t)n * j]);
        best = fmax(best, s);
    }
    red[threadIdx.x] = best;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + w]);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[b] = red[0];
}

// The powers of matrix b lie one after the other (Y^k at Q + (4 b + k - 1) nn), and
// so do its three phi-matrices (phi_k at P + (3 b + k) nn).
// T_k = sum_{j < 4} c_jk Y^j + (top: c_4k Y^4, else R_k), c_jk = 1 / (4 i + j + k)!
struct TaylorBlock {
    double c[5][3];
};
__global__ void k_taylor_block(int n, int64_t nn, bool top, TaylorBlock t, const double *Q, const double *R, double *T)
{
    const int b = blockIdx.y;
    const double *y = Q + 4 * b * nn;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nn; e += (int64_t)gridDim.x * blockDim.x) {
        const bool diag = e % n == e / n;
        const double y1 = y[e], y2 = y[nn + e], y3 = y[2 * nn + e], y4 = top ? y[3 * nn + e] : 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            double v = top ? t.c[4][k] * y4 : R[(3 * b + k) * nn + e];
            v = fma(t.c[3][k], y3, v);
            v = fma(t.c[2][k], y2, v);
            v = fma(t.c[1][k], y1, v);
            T[(3 * b + k) * nn + e] = diag ? v + t.c[0][k] : v;
        }
    }
}

// squaring update (T: phi_0 times the three)
__global__ void k_square_update(int64_t nn, const double *T, double *P)
{
    const int b = blockIdx.y;
    const double *t = T + 3 * b * nn;
    double *p = P + 3 * b * nn;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nn;
         e += (int64_t)gridDim.x * blockDim.x) {
        const double o1 = p[nn + e], o2 = p[2 * nn + e];
        p[e] = t[e];
        p[nn + e] = __dmul_rn(__dadd_rn(t[nn + e], o1), 0.5);
        p[2 * nn + e] = __dmul_rn(__dadd_rn(__dadd_rn(t[2 * nn + e], o1), o2), 0.25);
    }
}

__global__ void k_extract(int64_t nn, const double *const *src, double *const *dst)
{
    const int b = blockIdx.y;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nn;
         e += (int64_t)gridDim.x * blockDim.x)
        dst[b][e] = src[b][e];
}

// dst_b = lo_b - ell_b hi_b  (phi_{ell-1} - ell phi_ell)
__global__ void k_extract_deriv(int64_t nn, const double *const *lo, const double *const *hi,
                                const int *ell, double *const *dst)
{
    const int b = blockIdx.y;
    if (!dst[b]) return;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nn;
         e += (int64_t)gridDim.x * blockDim.x)
        dst[b][e] = lo[b][e] - (double)ell[b] * hi[b][e];
}

// C_b = A_b [B_b0 ... B_b(m-1)] for column-major n x n blocks, entries b of the
// batch sA, sB, sC apart, a right-hand entry's m blocks one after the other (and
// the products')
void batched_products(const mm::Context &ctx, int n, int m, int nb, const double *A, int64_t sA, const double *B,
                      int64_t sB, double *C, int64_t sC, cudaStream_t st)
{
    mm::Product p{};
    p.A = mm::matrix_view(n, A, 0);
    p.B = mm::matrix_view(n, B, 1);
    p.B.rows = (int64_t)m * n;
    p.A.batch = p.B.batch = nb;
    p.A.stride = sA;
    p.B.stride = sB;
    p.out = C;
    p.stride = sC;
    mm::run_products(ctx, &p, 1, st);
}
}  // namespace

ds_status phi_batch_f64(int n, const std::vector<PhiJob> &jobs, cudaStream_t st)
{
    const int nb = (int)jobs.size();
    if (nb == 0) return DS_OK;
    const int64_t nn = (int64_t)n * n, tot = nn * nb;
    // workspace: Y .. Y^4, phi0..2, their products (10 blocks), tables, digit images
    double *ws = nullptr;
    DS_CUDA_TRY(pool_alloc(&ws, sizeof(double) * tot * 10, st));
    double *Q = ws, *P = ws + 4 * tot, *T = ws + 7 * tot;
    mm::Context ctx;
    if (mm::use_digits(n, n, nb)) {
        mm::View v = mm::matrix_view(n, nullptr, 0);
        v.batch = nb;
        size_t bytes = mm::image_total(v, mm::kRowBlock);
        v.rows = 3 * (int64_t)n + 64;   // padded to whole column tiles
        bytes += mm::image_total(v, 1) + mm::kAlign + mm::left_bytes(n, 3 * n, nb);
        if (pool_alloc((void **)&ctx.ws, bytes, st) == cudaSuccess) {
            ctx.ws_bytes = bytes;
        } else {
            cudaGetLastError();   // short of memory: the FP64 pipe
            ctx.ws = nullptr;
        }
    }
    auto release = [&](void *tab) {
        cudaFreeAsync(ws, st);
        if (ctx.ws) cudaFreeAsync(ctx.ws, st);
        if (tab) cudaFreeAsync(tab, st);
    };

    std::vector<const double *> hA(nb);
    std::vector<double> hz(nb);
    for (int b = 0; b < nb; ++b) { hA[b] = jobs[b].A; hz[b] = jobs[b].z; }
    void *tab = nullptr;
    const size_t tab_bytes = sizeof(void *) * nb * 3 + sizeof(double) * nb * 2 + sizeof(int) * nb;
    cudaError_t e = pool_alloc(&tab, tab_bytes, st);
    if (e != cudaSuccess) { release(nullptr); return fail(DS_ERR_OOM, "phi table"); }
    const double **dA = (const double **)tab;
    double **dSrc = (double **)((char *)tab + sizeof(void *) * nb);
    double **dDst = (double **)((char *)tab + sizeof(void *) * nb * 2);
    double *dz = (double *)((char *)tab + sizeof(void *) * nb * 3);
    double *dnorm = dz + nb;
    int *ds_ = (int *)(dnorm + nb);
    cudaMemcpyAsync(dA, hA.data(), sizeof(void *) * nb, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(dz, hz.data(), sizeof(double) * nb, cudaMemcpyHostToDevice, st);

    dim3 g2((unsigned)std::min<int64_t>((nn + 255) / 256, 1024), nb);
    k_build_X<<<g2, 256, 0, st>>>(nn, dA, dz, Q, 4 * nn);
    k_norm1<<<nb, 256, 0, st>>>(n, Q, 4 * nn, dnorm);
    std::vector<double> hnorm(nb);
    cudaMemcpyAsync(hnorm.data(), dnorm, sizeof(double) * nb, cudaMemcpyDeviceToHost, st);
    DS_CUDA_TRY(cudaStreamSynchronize(st));
    std::vector<int> hs(nb);
    int smax = 0;
    for (int b = 0; b < nb; ++b) {
        if (!isfinite(hnorm[b])) {
            release(tab);
            return fail(DS_ERR_NONFINITE, "phi setup: non-finite matrix entry");
        }
        int s = 0;
        while (ldexp(hnorm[b], -s) > 0.5) ++s;
        hs[b] = s;
        smax = std::max(smax, s);
    }
    // the batch in order of falling s; Y = (2^-s z) A
    std::vector<int> perm(nb), sp(nb);
    for (int b = 0; b < nb; ++b) perm[b] = b;
    std::stable_sort(perm.begin(), perm.end(), [&](int x, int y) { return hs[x] > hs[y]; });
    for (int b = 0; b < nb; ++b) {
        sp[b] = hs[perm[b]];
        hA[b] = jobs[perm[b]].A;
        hz[b] = ldexp(jobs[perm[b]].z, -sp[b]);
    }
    cudaMemcpyAsync(dA, hA.data(), sizeof(void *) * nb, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(dz, hz.data(), sizeof(double) * nb, cudaMemcpyHostToDevice, st);
    k_build_X<<<g2, 256, 0, st>>>(nn, dA, dz, Q, 4 * nn);

    // Taylor: phi_k(Y) = sum_j Y^j / (j + k)!
    batched_products(ctx, n, 1, nb, Q, 4 * nn, Q, 4 * nn, Q + nn, 4 * nn, st);              // Y^2
    batched_products(ctx, n, 2, nb, Q + nn, 4 * nn, Q, 4 * nn, Q + 2 * nn, 4 * nn, st);     // Y^3, Y^4
    auto block = [](int i) {
        double fact[20] = {1.0};
        for (int j = 1; j < 20; ++j) fact[j] = fact[j - 1] * j;
        TaylorBlock t;
        for (int j = 0; j < 5; ++j)
            for (int k = 0; k < 3; ++k) t.c[j][k] = 1.0 / fact[4 * i + j + k];
        return t;
    };
    k_taylor_block<<<g2, 256, 0, st>>>(n, nn, true, block(3), Q, nullptr, P);
    for (int i = 2; i >= 0; --i) {
        batched_products(ctx, n, 3, nb, Q + 3 * nn, 4 * nn, P, 3 * nn, T, 3 * nn, st);
        k_taylor_block<<<g2, 256, 0, st>>>(n, nn, false, block(i), Q, T, P);
    }
    for (int it = 1; it <= smax; ++it) {
        int active = 0;
        while (active < nb && sp[active] >= it) ++active;
        batched_products(ctx, n, 3, active, P, 3 * nn, P, 3 * nn, T, 3 * nn, st);
        k_square_update<<<dim3(g2.x, active), 256, 0, st>>>(nn, T, P);
    }
    std::vector<double *> hsrc(nb), hdst(nb);
    for (int b = 0; b < nb; ++b) {
        const PhiJob &job = jobs[perm[b]];
        const int l = job.ell;
        hsrc[b] = P + (3 * b + l) * nn;
        hdst[b] = job.out;
    }
    cudaMemcpyAsync(dSrc, hsrc.data(), sizeof(void *) * nb, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(dDst, hdst.data(), sizeof(void *) * nb, cudaMemcpyHostToDevice, st);
    k_extract<<<g2, 256, 0, st>>>(nn, (const double *const *)dSrc, (double *const *)dDst);
    bool any_d = false;
    for (int b = 0; b < nb; ++b) any_d |= (jobs[b].dout != nullptr);
    if (any_d) {
        std::vector<double *> hlo(nb), hdd(nb);
        std::vector<int> hell(nb);
        for (int b = 0; b < nb; ++b) {
            const PhiJob &job = jobs[perm[b]];
            const int l = job.ell;
            hlo[b] = P + (3 * b + l - 1) * nn;
            hsrc[b] = P + (3 * b + l) * nn;
            hdd[b] = job.dout;
            hell[b] = l;
        }
        // the tables are reused: dA <- lo, dSrc <- hi, dDst <- dout, ds_ <- ell
        cudaMemcpyAsync(dA, hlo.data(), sizeof(void *) * nb, cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(dSrc, hsrc.data(), sizeof(void *) * nb, cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(dDst, hdd.data(), sizeof(void *) * nb, cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(ds_, hell.data(), sizeof(int) * nb, cudaMemcpyHostToDevice, st);
        k_extract_deriv<<<g2, 256, 0, st>>>(nn, (const double *const *)dA, (const double *const *)dSrc, ds_,
                                            (double *const *)dDst);
    }
    release(tab);
    DS_CUDA_TRY(cudaStreamSynchronize(st));
    DS_CUDA_TRY(cudaGetLastError());
    return DS_OK;
}

namespace {
// Aemb (2n x 2n, column-major) = [[zr A, -zi A], [zi A, zr A]]
__global__ void k_embed(int n, const double *__restrict__ A, double zr, double zi, double *__restrict__ E)
{
    const int64_t m = 2 * (int64_t)n, mm = m * m;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < mm;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e % m, c = e / m;
        const int64_t i = r % n, j = c % n;
        const double a = A[i + (int64_t)n * j];
        const bool lower = r >= n, right = c >= n;
        double v;
        if (lower == right) v = zr * a;        // diagonal blocks
        else if (lower) v = zi * a;            // bottom-left
        else v = -zi * a;                      // top-right
        E[e] = v;
    }
}
// re = top-left n x n block, im = bottom-left block of a 2n x 2n matrix
__global__ void k_unembed(int n, const double *__restrict__ E, double *__restrict__ re, double *__restrict__ im)
{
    const int64_t nn = (int64_t)n * n, m = 2 * (int64_t)n;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nn;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e % n, j = e / n;
        re[e] = E[i + m * j];
        im[e] = E[(i + n) + m * j];
    }
}
__global__ void k_fold_cplx(int64_t nn, const double *__restrict__ Qr, const double *__restrict__ Qi, double er,
                            double ei, double *__restrict__ M1, double *__restrict__ M2)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nn;
         e += (int64_t)gridDim.x * blockDim.x) {
        M1[e] = er * Qr[e] - ei * Qi[e];
        M2[e] = -(er * Qi[e] + ei * Qr[e]);
    }
}
}  // namespace

void launch_fold_cplx(int64_t nn, const double *Qr, const double *Qi, double er, double ei, double *M1,
                      double *M2, cudaStream_t st)
{
    k_fold_cplx<<<grid_for(nn), 256, 0, st>>>(nn, Qr, Qi, er, ei, M1, M2);
}

ds_status phi_batch_cplx(int n, const std::vector<PhiJobC> &jobs, cudaStream_t st)
{
    const int nb = (int)jobs.size();
    if (nb == 0) return DS_OK;
    const int64_t m = 2 * (int64_t)n, mm = m * m;
    double *buf = nullptr;
    DS_CUDA_TRY(pool_alloc(&buf, sizeof(double) * mm * nb * 2, st));
    double *emb = buf, *res = buf + mm * nb;
    std::vector<PhiJob> rj(nb);
    for (int b = 0; b < nb; ++b) {
        k_embed<<<grid_for(mm), 256, 0, st>>>(n, jobs[b].A, jobs[b].zr, jobs[b].zi, emb + b * mm);
        rj[b].A = emb + b * mm;
        rj[b].z = 1.0;
        rj[b].ell = jobs[b].ell;
        rj[b].out = res + b * mm;
        rj[b].dout = nullptr;
    }
    ds_status r = phi_batch_f64((int)m, rj, st);
    if (r != DS_OK) { cudaFreeAsync(buf, st); return r; }
    for (int b = 0; b < nb; ++b)
        k_unembed<<<grid_for((int64_t)n * n), 256, 0, st>>>(n, res + b * mm, jobs[b].out_re, jobs[b].out_im);
    cudaFreeAsync(buf, st);
    DS_CUDA_TRY(cudaStreamSynchronize(st));
    DS_CUDA_TRY(cudaGetLastError());
    return DS_OK;
}

}  // namespace ds
