// Krylov vector kernels: deterministic two-stage reductions (per-CTA partials,
// the last CTA to finish reduces them in a fixed order, so no extra launch and
// no run-to-run variation), the GMRES cycle's ends and the fused BiCGStab
// updates (the orthogonalisation is in ortho.cu).  Scalars never leave the device inside a step.
#include <cstdlib>
#include "krylov.cuh"

#include <cmath>

namespace {

constexpr int kVB = 256;  // block size of all streaming vector kernels

// Reduce NV per-thread values over the grid.  Returns true in every thread of
// the last CTA to finish; tot[] is then valid in thread 0 of that CTA.
template <int NV>
__device__ __forceinline__ bool grid_reduce(double (&v)[NV], double *__restrict__ part,
                                            unsigned *__restrict__ ticket, double (&tot)[NV]) {
    __shared__ double sh[32];
    __shared__ bool last;
    const int G = gridDim.x;
#pragma unroll
    for (int k = 0; k < NV; k++) {
        const double b = xbd::block_sum(v[k], sh);
        if (threadIdx.x == 0) part[k * G + blockIdx.x] = b;
    }
    if (threadIdx.x == 0) {
        __threadfence();
        last = (atomicAdd(ticket, 1u) == (unsigned)G - 1);
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
#pragma unroll
    for (int k = 0; k < NV; k++) {
        double a = 0.0;
        for (int i = threadIdx.x; i < G; i += blockDim.x) a += __ldcg(part + k * G + i);
        tot[k] = xbd::block_sum(a, sh);
    }
    if (threadIdx.x == 0) *ticket = 0u;
    return true;
}

__device__ __forceinline__ int64_t gtid() { return blockIdx.x * (int64_t)blockDim.x + threadIdx.x; }
__device__ __forceinline__ int64_t gstride() { return (int64_t)gridDim.x * blockDim.x; }

// ---- plain vector ops --------------------------------------------------------

__global__ void k_dot(int64_t n, const double *__restrict__ x, const double *__restrict__ y,
                      double *__restrict__ part, unsigned *__restrict__ ticket,
                      double *__restrict__ out, int sq, int vec) {
    double a0 = 0.0, a1 = 0.0;
    int64_t done = 0;
    if (vec) {
        const double2 *x2 = reinterpret_cast<const double2 *>(x);
        const double2 *y2 = reinterpret_cast<const double2 *>(y);
        const int64_t nv = n / 2;
        for (int64_t e = gtid(); e < nv; e += gstride()) {
            const double2 a = x2[e], b = y2[e];
            a0 = fma(a.x, b.x, a0);
            a1 = fma(a.y, b.y, a1);
        }
        done = nv * 2;
    }
    for (int64_t i = done + gtid(); i < n; i += gstride()) a0 = fma(x[i], y[i], a0);
    double v[1] = {a0 + a1};
    double t[1];
    if (grid_reduce<1>(v, part, ticket, t) && threadIdx.x == 0) *out = sq ? sqrt(t[0]) : t[0];
}

__global__ void k_axpy(int64_t n, double a, const double *__restrict__ x, double *__restrict__ y) {
    for (int64_t i = gtid(); i < n; i += gstride()) y[i] = fma(a, x[i], y[i]);
}
__global__ void k_copy(int64_t n, const double *__restrict__ x, double *__restrict__ y) {
    for (int64_t i = gtid(); i < n; i += gstride()) y[i] = x[i];
}
__global__ void k_scale(int64_t n, double a, double *__restrict__ x) {
    for (int64_t i = gtid(); i < n; i += gstride()) x[i] *= a;
}
__global__ void k_fill(int64_t n, double a, double *__restrict__ x) {
    for (int64_t i = gtid(); i < n; i += gstride()) x[i] = a;
}

// Grid of a streaming/reduction launch of kernel k over n elements: exactly the
// CTAs that fit on the GPU at once (fewer for small n), so a grid-stride pass
// runs as one coherent wave.
template <typename K>
int rgrid(K k, int64_t n) {
    return xb::resident_grid((const void *)k, kVB, n, 4);
}

// ---- GMRES ----------------------------------------------------------------------

// ||r0|| -> start a cycle: g = (beta, 0, ...), sc[0] = 1/beta.
template <typename VB>
__global__ void k_gm_init(int64_t n, const VB *__restrict__ r0, xb::GmDev st, double tau,
                          double *__restrict__ part, unsigned *__restrict__ ticket) {
    double v[1] = {0.0};
    for (int64_t i = gtid(); i < n; i += gstride()) {
        const double a = (double)r0[i];
        v[0] = fma(a, a, v[0]);
    }
    double t[1];
    if (grid_reduce<1>(v, part, ticket, t)) {
        for (int i = threadIdx.x; i <= st.M; i += blockDim.x) st.g[i] = 0.0;
        __syncthreads();
        if (threadIdx.x == 0) {
            const double beta = sqrt(t[0]);
            st.g[0] = beta;
            st.sc[0] = beta > 0.0 ? 1.0 / beta : 0.0;
            st.scf[0] = (float)st.sc[0];
            st.misc[xb::GM_BETA] = beta;
            const double bn = st.misc[xb::GM_BNORM];
            st.misc[xb::GM_RES] = bn > 0.0 ? beta / bn : 0.0;
            st.misc[xb::GM_K] = 0.0;
            st.misc[xb::GM_STOP] = 0.0;
            st.misc[xb::GM_TAU] = tau;
            st.misc[xb::GM_LEN2] = 0.0;
            st.misc[xb::GM_RAW] = 0.0;
        }
    }
}

template <typename VB>
struct V16;
template <>
struct V16<double> {
    using T = double2;
    static constexpr int N = 2;
    __device__ static double get(const double2 &v, int k) { return k == 0 ? v.x : v.y; }
    __device__ static void set(double2 &v, int k, double a) {
        if (k == 0) v.x = a;
        else v.y = a;
    }
};
template <>
struct V16<float> {
    using T = float4;
    static constexpr int N = 4;
    __device__ static float get(const float4 &v, int k) {
        return k == 0 ? v.x : (k == 1 ? v.y : (k == 2 ? v.z : v.w));
    }
    __device__ static void set(float4 &v, int k, float a) {
        if (k == 0) v.x = a;
        else if (k == 1) v.y = a;
        else if (k == 2) v.z = a;
        else v.w = a;
    }
};

// Least squares R y = g (upper triangular k x k), then y_i *= sc[i].  One CTA:
// the triangle comes into shared memory together (k <= kSolveK), then warp 0
// solves by columns; y_i = s_i / r_ii is a product with the reciprocal taken
// beforehand and one correction step, as accurate as the division and a third
// of its latency.
constexpr int kSolveK = 64;
__global__ void __launch_bounds__(256) k_gm_solve(xb::GmDev st) {
    __shared__ double R[kSolveK][kSolveK + 1], s[512], rinv[512];
    const int k = (int)st.misc[xb::GM_K];
    const int tid = threadIdx.x;
    const size_t ldh = st.M + 1;
    const bool held = k <= kSolveK;
    if (held)
        for (int t = tid; t < k * k; t += blockDim.x) {
            const int c = t / k, r = t % k;
            if (r <= c) R[c][r] = st.H[c * ldh + r];
        }
    for (int i = tid; i < k; i += blockDim.x) {
        s[i] = st.g[i];
        rinv[i] = 1.0 / st.H[i * ldh + i];
    }
    __syncthreads();
    if (tid >= 32) return;
    for (int i = k - 1; i >= 0; i--) {
        const double *col = held ? R[i] : st.H + i * ldh;
        const double d = col[i], si = s[i];
        double y = si * rinv[i];
        if (fabs(d) > 1e-280 && fabs(d) < 1e280) y = fma(fma(-y, d, si), rinv[i], y);
        else y = si / d;
        for (int r = tid; r < i; r += 32) s[r] = fma(-col[r], y, s[r]);
        if (tid == 0) st.y[i] = y * st.sc[i];
        __syncwarp();
    }
}

// x += sum_i y_i V_i (each basis vector read once; 16-byte vectors when the
// basis and x are aligned).
template <typename VB, typename VX>
__global__ void __launch_bounds__(kVB) k_gm_xupd(int64_t n, const VB *__restrict__ V, int64_t ld,
                                                 xb::GmDev st, VX *__restrict__ x, int vec) {
    __shared__ double ys[512];
    const int k = (int)st.misc[xb::GM_K];
    for (int i = threadIdx.x; i < k && i < 512; i += blockDim.x) ys[i] = st.y[i];
    __syncthreads();
    int64_t done = 0;
    if (vec) {
        using T = typename V16<VB>::T;
        using TX = typename V16<VX>::T;
        constexpr int N = V16<VB>::N;
        static_assert(V16<VB>::N == V16<VX>::N, "same width");
        const int64_t nv = n / N;
        for (int64_t e = gtid(); e < nv; e += gstride()) {
            VX s[N];
#pragma unroll
            for (int q = 0; q < N; q++) s[q] = VX(0);
            for (int i = 0; i < k; i++) {
                const T v = reinterpret_cast<const T *>(V + (size_t)i * ld)[e];
                const VX yi = (VX)ys[i];
#pragma unroll
                for (int q = 0; q < N; q++) s[q] = fma(yi, (VX)V16<VB>::get(v, q), s[q]);
            }
            TX a = reinterpret_cast<TX *>(x)[e];
#pragma unroll
            for (int q = 0; q < N; q++) V16<VX>::set(a, q, V16<VX>::get(a, q) + s[q]);
            reinterpret_cast<TX *>(x)[e] = a;
        }
        done = nv * N;
    }
    for (int64_t e = done + gtid(); e < n; e += gstride()) {
        VX s = VX(0);
        for (int i = 0; i < k; i++) s = fma((VX)ys[i], (VX)V[(size_t)i * ld + e], s);
        x[e] += s;
    }
}

// ---- BiCGStab ------------------------------------------------------------------
// Every kernel walks its vectors as 16-byte pairs when all of them are 16-byte
// aligned (vec != 0), then finishes the odd tail element by element.

__device__ __forceinline__ double2 ld2(const double *a, int64_t i) {
    return reinterpret_cast<const double2 *>(a)[i];
}
__device__ __forceinline__ void st2(double *a, int64_t i, double2 v) {
    reinterpret_cast<double2 *>(a)[i] = v;
}

// rho = (rhat, r) with rhat = r at a (re)start; alpha = omega = rho_old = 1.
__global__ void k_bi_init(int64_t n, const double *__restrict__ r, double *__restrict__ sc,
                          double tau2, double *__restrict__ part, unsigned *__restrict__ ticket,
                          int vec) {
    double v[1] = {0.0};
    int64_t done = 0;
    if (vec) {
        for (int64_t i = gtid(); i < n / 2; i += gstride()) {
            const double2 a = ld2(r, i);
            v[0] = fma(a.y, a.y, fma(a.x, a.x, v[0]));
        }
        done = n / 2 * 2;
    }
    for (int64_t i = done + gtid(); i < n; i += gstride()) v[0] = fma(r[i], r[i], v[0]);
    double t[1];
    if (grid_reduce<1>(v, part, ticket, t) && threadIdx.x == 0) {
        sc[xb::BI_RHO] = t[0];
        sc[xb::BI_RHO_OLD] = 1.0;
        sc[xb::BI_ALPHA] = 1.0;
        sc[xb::BI_OMEGA] = 1.0;
        sc[xb::BI_RNORM2] = t[0];
        sc[xb::BI_SNORM2] = INFINITY;
        sc[xb::BI_FLAG] = 0.0;
        sc[xb::BI_TAU2] = tau2;
    }
}

// p = r + beta (p - omega v), beta = (rho/rho_old)(alpha/omega).
__global__ void k_bi_p(int64_t n, const double *__restrict__ sc, const double *__restrict__ r,
                       double *__restrict__ p, const double *__restrict__ v, int vec) {
    if (sc[xb::BI_FLAG] != 0.0) return;
    const double beta =
        (sc[xb::BI_RHO] / sc[xb::BI_RHO_OLD]) * (sc[xb::BI_ALPHA] / sc[xb::BI_OMEGA]);
    const double om = sc[xb::BI_OMEGA];
    auto f = [=](double ri, double pi, double vi) { return fma(beta, fma(-om, vi, pi), ri); };
    int64_t done = 0;
    if (vec) {
        for (int64_t i = gtid(); i < n / 2; i += gstride()) {
            const double2 a = ld2(r, i), c = ld2(v, i);
            double2 q = ld2(p, i);
            q.x = f(a.x, q.x, c.x);
            q.y = f(a.y, q.y, c.y);
            st2(p, i, q);
        }
        done = n / 2 * 2;
    }
    for (int64_t i = done + gtid(); i < n; i += gstride()) p[i] = f(r[i], p[i], v[i]);
}

// sigma = (rhat, v); alpha = rho / sigma.
__global__ void k_bi_sigma(int64_t n, double *__restrict__ sc, const double *__restrict__ rh,
                           const double *__restrict__ v, double *__restrict__ part,
                           unsigned *__restrict__ ticket, int vec) {
    if (sc[xb::BI_FLAG] != 0.0) return;
    double a[1] = {0.0};
    int64_t done = 0;
    if (vec) {
        for (int64_t i = gtid(); i < n / 2; i += gstride()) {
            const double2 h = ld2(rh, i), w = ld2(v, i);
            a[0] = fma(h.y, w.y, fma(h.x, w.x, a[0]));
        }
        done = n / 2 * 2;
    }
    for (int64_t i = done + gtid(); i < n; i += gstride()) a[0] = fma(rh[i], v[i], a[0]);
    double t[1];
    if (grid_reduce<1>(a, part, ticket, t) && threadIdx.x == 0) {
        if (t[0] == 0.0) sc[xb::BI_FLAG] = 3.0;
        else sc[xb::BI_ALPHA] = sc[xb::BI_RHO] / t[0];
    }
}

// s = r - alpha v, ||s||^2.
__global__ void k_bi_s(int64_t n, double *__restrict__ sc, const double *__restrict__ r,
                       const double *__restrict__ v, double *__restrict__ s,
                       double *__restrict__ part, unsigned *__restrict__ ticket, int vec) {
    if (sc[xb::BI_FLAG] != 0.0) return;
    const double al = sc[xb::BI_ALPHA];
    double a[1] = {0.0};
    int64_t done = 0;
    if (vec) {
        for (int64_t i = gtid(); i < n / 2; i += gstride()) {
            const double2 q = ld2(r, i), w = ld2(v, i);
            double2 si;
            si.x = fma(-al, w.x, q.x);
            si.y = fma(-al, w.y, q.y);
            st2(s, i, si);
            a[0] = fma(si.y, si.y, fma(si.x, si.x, a[0]));
        }
        done = n / 2 * 2;
    }
    for (int64_t i = done + gtid(); i < n; i += gstride()) {
        const double si = fma(-al, v[i], r[i]);
        s[i] = si;
        a[0] = fma(si, si, a[0]);
    }
    double t[1];
    if (grid_reduce<1>(a, part, ticket, t) && threadIdx.x == 0) sc[xb::BI_SNORM2] = t[0];
}

// omega = (t, s) / (t, t).
__global__ void k_bi_omega(int64_t n, double *__restrict__ sc, const double *__restrict__ t,
                           const double *__restrict__ s, double *__restrict__ part,
                           unsigned *__restrict__ ticket, int vec) {
    if (sc[xb::BI_FLAG] != 0.0) return;
    double a[2] = {0.0, 0.0};
    int64_t done = 0;
    if (vec) {
        for (int64_t i = gtid(); i < n / 2; i += gstride()) {
            const double2 u = ld2(t, i), w = ld2(s, i);
            a[0] = fma(u.y, w.y, fma(u.x, w.x, a[0]));
            a[1] = fma(u.y, u.y, fma(u.x, u.x, a[1]));
        }
        done = n / 2 * 2;
    }
    for (int64_t i = done + gtid(); i < n; i += gstride()) {
        a[0] = fma(t[i], s[i], a[0]);
        a[1] = fma(t[i], t[i], a[1]);
    }
    double tt[2];
    if (grid_reduce<2>(a, part, ticket, tt) && threadIdx.x == 0) {
        if (sc[xb::BI_SNORM2] <= sc[xb::BI_TAU2]) return;  // s already converged
        if (tt[1] == 0.0) sc[xb::BI_FLAG] = 4.0;
        else sc[xb::BI_OMEGA] = tt[0] / tt[1];
    }
}

// x += alpha p + omega sx;  r = s - omega t;  ||r||^2, rho_next = (rhat, r).
// sx is s itself, or M^{-1} s (and p is M^{-1} p) under right preconditioning.
// When ||s|| already met the threshold: x += alpha p only, flag = 1 (done).
__global__ void k_bi_xr(int64_t n, double *__restrict__ sc, double *__restrict__ x,
                        const double *__restrict__ p, const double *__restrict__ s,
                        const double *sx, const double *__restrict__ t,
                        double *__restrict__ r, const double *__restrict__ rh,
                        double *__restrict__ part, unsigned *__restrict__ ticket, int vec) {
    if (sc[xb::BI_FLAG] != 0.0) return;
    const double al = sc[xb::BI_ALPHA];
    if (sc[xb::BI_SNORM2] <= sc[xb::BI_TAU2]) {
        for (int64_t i = gtid(); i < n; i += gstride()) x[i] = fma(al, p[i], x[i]);
        double a[1] = {0.0}, tt[1];
        if (grid_reduce<1>(a, part, ticket, tt) && threadIdx.x == 0) {
            sc[xb::BI_RNORM2] = sc[xb::BI_SNORM2];
            sc[xb::BI_FLAG] = 1.0;
        }
        return;
    }
    const double om = sc[xb::BI_OMEGA];
    double a[2] = {0.0, 0.0};
    auto f = [&](double &xi, double pi, double si, double sxi, double ti, double hi) {
        xi = fma(om, sxi, fma(al, pi, xi));
        const double ri = fma(-om, ti, si);
        a[0] = fma(ri, ri, a[0]);
        a[1] = fma(hi, ri, a[1]);
        return ri;
    };
    int64_t done = 0;
    if (vec) {
        for (int64_t i = gtid(); i < n / 2; i += gstride()) {
            double2 xv = ld2(x, i), rv;
            const double2 pv = ld2(p, i), sv = ld2(s, i), tv = ld2(t, i), hv = ld2(rh, i);
            const double2 zv = ld2(sx, i);
            rv.x = f(xv.x, pv.x, sv.x, zv.x, tv.x, hv.x);
            rv.y = f(xv.y, pv.y, sv.y, zv.y, tv.y, hv.y);
            st2(x, i, xv);
            st2(r, i, rv);
        }
        done = n / 2 * 2;
    }
    for (int64_t i = done + gtid(); i < n; i += gstride()) {
        double xi = x[i];
        r[i] = f(xi, p[i], s[i], sx[i], t[i], rh[i]);
        x[i] = xi;
    }
    double tt[2];
    if (grid_reduce<2>(a, part, ticket, tt) && threadIdx.x == 0) {
        sc[xb::BI_RNORM2] = tt[0];
        sc[xb::BI_RHO_OLD] = sc[xb::BI_RHO];
        sc[xb::BI_RHO] = tt[1];
        if (tt[0] <= sc[xb::BI_TAU2]) sc[xb::BI_FLAG] = 1.0;
        else if (tt[1] == 0.0) sc[xb::BI_FLAG] = 2.0;
        else if (om == 0.0) sc[xb::BI_FLAG] = 5.0;
    }
}

// ---- mixed precision helpers ------------------------------------------------------

__global__ void k_cast_scaled(int64_t n, const double *__restrict__ a,
                              const double *__restrict__ scale, float *__restrict__ b) {
    const double s = *scale;
    const double inv = s > 0.0 ? 1.0 / s : 0.0;
    for (int64_t i = gtid(); i < n; i += gstride()) b[i] = (float)(a[i] * inv);
}

__global__ void k_add_scaled(int64_t n, double *__restrict__ x, const double *__restrict__ scale,
                             const float *__restrict__ d) {
    const double s = *scale;
    for (int64_t i = gtid(); i < n; i += gstride()) x[i] = fma(s, (double)d[i], x[i]);
}

}  // namespace

namespace xb {

GmDev gm_layout(double *base, int M) {
    GmDev st;
    st.M = M;
    double *q = base;
    st.H = q; q += (size_t)(M + 1) * M;
    st.cs = q; q += M;
    st.sn = q; q += M;
    st.g = q; q += M + 1;
    st.sc = q; q += M + 1;
    st.y = q; q += M;
    st.gram = q; q += 8 * (size_t)(M + 1);
    st.misc = q; q += GM_NMISC;
    st.scf = reinterpret_cast<float *>(q);
    return st;
}

int vdot(xb_plan *p, int64_t n, const double *x, const double *y, double *out, cudaStream_t s) {
    const int g = rgrid(k_dot, n);
    const int vec = (((uintptr_t)x | (uintptr_t)y) % 16) == 0 ? 1 : 0;
    k_dot<<<g, kVB, 0, s>>>(n, x, y, p->d_part, p->d_ticket, out, 0, vec);
    XB_LAUNCHED("k_dot");
    return XB_OK;
}
int vnrm2(xb_plan *p, int64_t n, const double *x, double *out, cudaStream_t s) {
    const int g = rgrid(k_dot, n);
    const int vec = ((uintptr_t)x % 16) == 0 ? 1 : 0;
    k_dot<<<g, kVB, 0, s>>>(n, x, x, p->d_part, p->d_ticket, out, 1, vec);
    XB_LAUNCHED("k_nrm2");
    return XB_OK;
}
int vaxpy(int64_t n, double a, const double *x, double *y, cudaStream_t s) {
    if (n <= 0) return XB_OK;
    k_axpy<<<rgrid(k_axpy, n), kVB, 0, s>>>(n, a, x, y);
    XB_LAUNCHED("k_axpy");
    return XB_OK;
}
int vcopy(int64_t n, const double *x, double *y, cudaStream_t s) {
    if (n <= 0) return XB_OK;
    k_copy<<<rgrid(k_copy, n), kVB, 0, s>>>(n, x, y);
    XB_LAUNCHED("k_copy");
    return XB_OK;
}
int vscale(int64_t n, double a, double *x, cudaStream_t s) {
    if (n <= 0) return XB_OK;
    k_scale<<<rgrid(k_scale, n), kVB, 0, s>>>(n, a, x);
    XB_LAUNCHED("k_scale");
    return XB_OK;
}
int vfill(int64_t n, double a, double *x, cudaStream_t s) {
    if (n <= 0) return XB_OK;
    k_fill<<<rgrid(k_fill, n), kVB, 0, s>>>(n, a, x);
    XB_LAUNCHED("k_fill");
    return XB_OK;
}

int gm_cycle_init(xb_plan *p, GmDev st, int64_t n, const double *r0, double tau, cudaStream_t s) {
    k_gm_init<double><<<rgrid(k_gm_init<double>, n), kVB, 0, s>>>(n, r0, st, tau, p->d_part,
                                                                 p->d_ticket);
    XB_LAUNCHED("k_gm_init");
    return XB_OK;
}
int gm_cycle_init_f32(xb_plan *p, GmDev st, int64_t n, const float *r0, double tau,
                      cudaStream_t s) {
    k_gm_init<float><<<rgrid(k_gm_init<float>, n), kVB, 0, s>>>(n, r0, st, tau, p->d_part,
                                                               p->d_ticket);
    XB_LAUNCHED("k_gm_init_f32");
    return XB_OK;
}

double ortho_passes(int ortho, int j, int kb, bool held) {
    const int k = j + 1, nb = (k + kb - 1) / kb, rounds = ortho == XB_ORTHO_DGKS ? 2 : 1;
    const double rows = 2.0 * rounds * k;
    if (held) return rows + 2.0;
    if (ortho == XB_ORTHO_MGS || ortho == XB_ORTHO_BCGS) return rows + 2.0 * nb + 1.0;
    return rows + rounds * (nb + 1.0) + 1.0;
}

int ortho_choice(int ortho, double tol, bool faulted) {
    if (ortho != XB_ORTHO_AUTO) return ortho;
    if (faulted) return XB_ORTHO_DGKS;
    return tol <= 1e-10 ? XB_ORTHO_MGS : XB_ORTHO_BCGS;
}

template <typename VB, typename VX>
int gm_update(xb_plan *p, GmDev st, int64_t n, const VB *V, int64_t ld, int k, VX *x,
              cudaStream_t s) {
    (void)p;
    (void)k;
    k_gm_solve<<<1, 256, 0, s>>>(st);
    XB_LAUNCHED("k_gm_solve");
    const int vec = (((uintptr_t)V % 16) == 0 && ((uintptr_t)x % 16) == 0 &&
                     ((ld * sizeof(VB)) % 16) == 0) ? 1 : 0;
    k_gm_xupd<VB, VX><<<rgrid(k_gm_xupd<VB, VX>, n), kVB, 0, s>>>(n, V, ld, st, x, vec);
    XB_LAUNCHED("k_gm_xupd");
    return XB_OK;
}
template int gm_update<double, double>(xb_plan *, GmDev, int64_t, const double *, int64_t, int,
                                       double *, cudaStream_t);
template int gm_update<float, float>(xb_plan *, GmDev, int64_t, const float *, int64_t, int,
                                     float *, cudaStream_t);

static int al16(const void *a) { return ((uintptr_t)a % 16) == 0; }

int bi_init(xb_plan *p, double *scal, int64_t n, const double *r, double tau2, cudaStream_t s) {
    k_bi_init<<<rgrid(k_bi_init, n), kVB, 0, s>>>(n, r, scal, tau2, p->d_part, p->d_ticket,
                                                  al16(r));
    XB_LAUNCHED("k_bi_init");
    return XB_OK;
}
int bi_p_update(double *scal, int64_t n, const double *r, double *pv, const double *v,
                cudaStream_t s) {
    k_bi_p<<<rgrid(k_bi_p, n), kVB, 0, s>>>(n, scal, r, pv, v, al16(r) & al16(pv) & al16(v));
    XB_LAUNCHED("k_bi_p");
    return XB_OK;
}
int bi_sigma(xb_plan *p, double *scal, int64_t n, const double *rh, const double *v,
             cudaStream_t s) {
    k_bi_sigma<<<rgrid(k_bi_sigma, n), kVB, 0, s>>>(n, scal, rh, v, p->d_part, p->d_ticket,
                                                   al16(rh) & al16(v));
    XB_LAUNCHED("k_bi_sigma");
    return XB_OK;
}
int bi_s_update(xb_plan *p, double *scal, int64_t n, const double *r, const double *v, double *sv,
                cudaStream_t s) {
    k_bi_s<<<rgrid(k_bi_s, n), kVB, 0, s>>>(n, scal, r, v, sv, p->d_part, p->d_ticket,
                                               al16(r) & al16(v) & al16(sv));
    XB_LAUNCHED("k_bi_s");
    return XB_OK;
}
int bi_omega(xb_plan *p, double *scal, int64_t n, const double *t, const double *sv,
             cudaStream_t s) {
    k_bi_omega<<<rgrid(k_bi_omega, n), kVB, 0, s>>>(n, scal, t, sv, p->d_part, p->d_ticket,
                                                   al16(t) & al16(sv));
    XB_LAUNCHED("k_bi_omega");
    return XB_OK;
}
int bi_xr_update(xb_plan *p, double *scal, int64_t n, double *x, const double *pv,
                 const double *sv, const double *sx, const double *t, double *r, const double *rh,
                 cudaStream_t s) {
    const int vec = al16(x) & al16(pv) & al16(sv) & al16(sx) & al16(t) & al16(r) & al16(rh);
    k_bi_xr<<<rgrid(k_bi_xr, n), kVB, 0, s>>>(n, scal, x, pv, sv, sx, t, r, rh, p->d_part,
                                                p->d_ticket, vec);
    XB_LAUNCHED("k_bi_xr");
    return XB_OK;
}

// r = b - A x
int residual(xb_plan *p, const double *b, const double *x, double *r, cudaStream_t s) {
    XB_TRY(vcopy(p->n, b, r, s));
    return spmv_launch(p, XB_VAR_AUTO, 0, 0, -1.0, x, 1.0, r, s);
}

int cast_f64_to_f32_scaled(int64_t n, const double *a, const double *scale_dev, float *b,
                           cudaStream_t s) {
    if (n <= 0) return XB_OK;
    k_cast_scaled<<<rgrid(k_cast_scaled, n), kVB, 0, s>>>(n, a, scale_dev, b);
    XB_LAUNCHED("k_cast_scaled");
    return XB_OK;
}

int add_scaled_f32(int64_t n, double *x, const double *scale_dev, const float *d, cudaStream_t s) {
    if (n <= 0) return XB_OK;
    k_add_scaled<<<rgrid(k_add_scaled, n), kVB, 0, s>>>(n, x, scale_dev, d);
    XB_LAUNCHED("k_add_scaled");
    return XB_OK;
}

}  // namespace xb
