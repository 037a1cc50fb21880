// Batched solve of many independent systems in ONE persistent kernel launch,
// captured in a CUDA graph and replayed.
//
// The launch is a grid of 8-CTA thread-block clusters, fed by two atomic
// queues (each ordered largest first):
//   - a large system (split_systems) is solved by a whole cluster: every CTA
//     owns a slice of the rows, dot products are combined across the cluster
//     through distributed shared memory (every CTA sums the 8 partials in rank
//     order, so all CTAs hold identical values), and hardware cluster
//     barriers order the shared vectors; a cluster's leader pulls these;
//   - smaller systems are pulled by each CTA on its own, as soon as it is
//     free, and solved with block-level reductions only.
// Most clusters take the cluster queue first and then the other; the first
// few start on the single-CTA queue and join the cluster queue after it.
// Every cluster barrier sits on a path whose branch conditions are
// cluster-uniform (iteration counts, reduced values, and a time-budget flag
// that rank 0 decides and broadcasts through a reduction), so all CTAs of a
// cluster reach the same barriers in the same order.
//
// The solver is restarted GMRES(m) with modified Gram-Schmidt or blocked
// classical Gram-Schmidt, both over blocks of 4 basis vectors (one pass, which
// applies the previous block's projection, and one four-value reduction per
// block; for MGS the block's dots are corrected by its own inner products, or,
// with many rows a CTA, taken a vector at a time), Givens least squares, the true-residual check at every restart (fault
// convergence narrows the implicit threshold), and, when enabled, the
// MM-ratio restart rule of Eq. (1) / Fig. 2 / Sec. 4.3 (m grows by 5, up to
// m_max, when 5 consecutive restart residuals change by less than theta).
#include "common.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <numeric>

namespace cg = cooperative_groups;

namespace {
constexpr int kCl = 8;          // CTAs per cluster
constexpr int kBT = 512;        // threads per CTA
constexpr int kLargeN = 30000;  // systems this large are always solved by a whole cluster
constexpr int kTile = 256;      // mode 1: entries a warp sums at a time, 8 a lane
}  // namespace

struct xb_batch_dev {
    int n, nnz, m, m_max, mode, zero_x, coop;
    int single;  // MGS a vector at a time (single_dots)
    int64_t ld;
    const int *rowptr, *col;
    const double *val, *b;
    double *x;
    double *V;  // (m_max+1) * ld basis
    double *H;  // per cooperating CTA: (m_max+1) * m_max Hessenberg (column-major)
    // mode 1: tiles of kTile entries of each CTA's part of the rows; part c has
    // tiles tptr[c] .. tptr[c + 1]
    int tptr[kCl + 1];
    const int *trow;  // row of a tile's first entry
    int *tinfo;       // row that a tile ends but does not start; -2: none, -1: ends no row
    double2 *tsum;    // sums of that row's entries in the tile, and of the entries after the last end
};

struct xb_batch {
    int count = 0;
    xb_batch_dev *d_sys = nullptr;
    xb_batch_info *d_info = nullptr;
    int *d_order = nullptr, *d_queue = nullptr;
    double *d_ws = nullptr;
    void *d_tiles = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    int grid = 0;
};

namespace {

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

constexpr int kNW = kBT / 32;

struct Smem {
    double part[2][4][kNW], slot[2][4], tot[2][4];   // sums of up to 4 values, two phases
    double g[XB_BATCH_MAX_M + 1], cs[XB_BATCH_MAX_M], sn[XB_BATCH_MAX_M], yv[XB_BATCH_MAX_M];
    double hc[XB_BATCH_MAX_M + 2];                   // the step's Hessenberg column, unrotated
    double hn[XB_BATCH_MAX_M + 1], sc[XB_BATCH_MAX_M + 1];  // norms of the stored basis vectors, 1 / them
    double sg[(XB_BATCH_MAX_M + 1) * 4];             // sc_i^2 (V_i, V_k), k in i's block of 4 before i
    double tt, len2;
    unsigned long long t_start;
    int q;
    int flag;
};

// The solve's view of the work: rows [r0, r1) of this CTA, and whether the
// CTAs of the cluster cooperate on this system.
struct Part {
    int r0, r1, coop, phase;
};

// Sums of NV <= 4 values over all cooperating CTAs, in a fixed order.  Every
// warp adds its lanes' values (four in a transposed tree: 6 adds instead of 20;
// an FP64 add holds a quarter of the SM for ~80 cycles whatever it adds), warp 0
// the warps' sums and, for a cluster, the 8 CTAs' after one cluster barrier.
// `while_w2` runs in warp 2 beside warp 0's sums, `fin` in warp 0 with value
// lane >> 3 of the total in every lane; then the CTA meets.  Slots of two phases
// alternate, so a slot is rewritten only after every CTA has passed the barrier
// of the sum that follows its last read.  The cluster barrier (or the CTA's)
// also orders the vectors written before it.
template <int NV, typename W2, typename Fin>
__device__ __forceinline__ void sums(const double (&v)[NV], Smem &S, Part &P, W2 while_w2, Fin fin) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, ph = P.phase;
    double k;
    if constexpr (NV == 4) {
        const bool h16 = lane & 16, h8 = lane & 8;
        double k0 = h16 ? v[2] : v[0], k1 = h16 ? v[3] : v[1];
        const double s0 = h16 ? v[0] : v[2], s1 = h16 ? v[1] : v[3];
        k0 += __shfl_xor_sync(0xffffffffu, s0, 16);
        k1 += __shfl_xor_sync(0xffffffffu, s1, 16);
        k = h8 ? k1 : k0;
        k += __shfl_xor_sync(0xffffffffu, h8 ? k0 : k1, 8);
    } else {
        k = v[0];
        k += __shfl_xor_sync(0xffffffffu, k, 16);
        k += __shfl_xor_sync(0xffffffffu, k, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
    if ((lane & 7) == 0 && (lane >> 3) < NV) S.part[ph][lane >> 3][w] = k;
    __syncthreads();
    const int q = lane >> 3, r = lane & 7;
    double a = 0.0;
    if (w == 0) {
        if (q < NV) a = S.part[ph][q][r] + S.part[ph][q][r + 8];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (P.coop && r == 0) S.slot[ph][q] = a;
    } else if (w == 2) {
        while_w2();
    }
    if (P.coop) {
        cg::cluster_group cl = cg::this_cluster();
        cl.sync();
        if (w == 0) {
            a = cl.map_shared_rank(&S.slot[0][0], r)[ph * 4 + q];
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        }
    }
    if (w == 0) {
        fin(a);
        if (r == 0) S.tot[ph][q] = a;
    }
    __syncthreads();
    P.phase ^= 1;
}

// The plain sum of one value, the same in every thread.
__device__ double coop_sum(double v, Smem &S, Part &P) {
    const double v1[1] = {v};
    const int ph = P.phase;
    sums<1>(v1, S, P, [] {}, [](double &) {});
    return S.tot[ph][0];
}

// Make every cooperating CTA's writes to the shared vectors visible to all.
__device__ __forceinline__ void coop_barrier(const Part &P) {
    if (P.coop) cg::this_cluster().sync();
    else __syncthreads();
}

// y[r0:r1] = alpha*A[r0:r1,:]*x (+ beta*y), beta 0 or 1.  x is written by the other CTAs
// of the cluster during the launch and ordered by the barrier (release / acquire)
// that follows: never the read-only path.
//   mode 0: one thread per row, x read at L2 (ld.global.cg), which leaves the L1
//           to the rows' entries (512 systems, power-law rows among them: 15.0 s,
//           16.0 through the L1; 48 systems 21.6 and 21.4 ms);
//   mode 1: part_tiles.
// Every row's sum has one fixed order, so results do not depend on scheduling.
__device__ __forceinline__ double row_dot(const int *__restrict__ col,
                                          const double *__restrict__ val, const double *x,
                                          int ka, int kb) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    int k = ka;
    for (; k + 3 < kb; k += 4) {  // four gathers in flight
        const int c0 = __ldg(col + k), c1 = __ldg(col + k + 1), c2 = __ldg(col + k + 2), c3 = __ldg(col + k + 3);
        const double v0 = __ldg(val + k), v1 = __ldg(val + k + 1), v2 = __ldg(val + k + 2), v3 = __ldg(val + k + 3);
        s0 = fma(v0, __ldcg(x + c0), s0);
        s1 = fma(v1, __ldcg(x + c1), s1);
        s2 = fma(v2, __ldcg(x + c2), s2);
        s3 = fma(v3, __ldcg(x + c3), s3);
    }
    for (; k < kb; k++) s0 = fma(__ldg(val + k), __ldcg(x + __ldg(col + k)), s0);
    return (s0 + s1) + (s2 + s3);
}

// A warp's shared memory in mode 1: the tile's values and gathered x, 8 entries
// and a gap for each lane (no bank conflicts), and the marks of row ends.
struct TileBuf {
    double2 vx[kTile + kTile / 8];
    unsigned char end[kTile];
};

// Mode 1: the CTA's entries in tiles of 256, whatever their rows.  A power law's
// rows differ by orders of magnitude, and an FP64 instruction holds a quarter of
// the SM for ~64 cycles however few lanes need it, so a lane sums 8 consecutive
// entries (8 FMAs for 256 of them), a segmented scan, ended by a vote, carries the
// sums of rows over lanes, and rows that leave their tile are completed after the
// CTA has met.  Loads of col and val cover whole sectors; the next tile's are on
// their way during the sums.  n = 40,900, 522,000 non-zeros, GMRES(30) on 8 CTAs:
// 133 us a step, 203 with a lane for a row of up to 32 entries and a warp for
// longer ones, 193 with 8 lanes for a row.
__device__ void part_tiles(const xb_batch_dev &D, const Part &P, int part, TileBuf *buf, double alpha,
                           const double *x, double beta, double *y) {
    const int *__restrict__ rp = D.rowptr;
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    TileBuf &B = buf[threadIdx.x >> 5];
    const int t0 = D.tptr[part], t1 = D.tptr[part + 1];
    if (t0 == t1) {
        if (beta == 0.0)
            for (int r = P.r0 + threadIdx.x; r < P.r1; r += blockDim.x) y[r] = 0.0;
        return;
    }
    const int e0 = __ldg(rp + P.r0), e1 = __ldg(rp + P.r1);
    int c[8];
    double v[8];
    auto load = [&](int t) {
        const unsigned at = (unsigned)e0 + (unsigned)(t - t0) * kTile + lane;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const bool in = t < t1 && at + 32 * i < (unsigned)e1;
            c[i] = in ? __ldg(D.col + at + 32 * i) : -1;
            v[i] = in ? __ldg(D.val + at + 32 * i) : 0.0;
        }
    };
    int t = t0 + (threadIdx.x >> 5);
    load(t);
    for (; t < t1; t += nw) {
        const int tb = e0 + (t - t0) * kTile, te = e1 - tb > kTile ? tb + kTile : e1;
        const int ra = t == t0 ? P.r0 : __ldg(D.trow + t), rb = t + 1 < t1 ? __ldg(D.trow + t + 1) + 1 : P.r1;
        double xv[8];
#pragma unroll
        for (int i = 0; i < 8; i++) xv[i] = c[i] >= 0 ? x[c[i]] : 0.0;
        reinterpret_cast<uint2 *>(B.end)[lane] = make_uint2(0, 0);
        __syncwarp();
        // the first 32 rows' bounds stay in registers
        const int fs = ra + lane < rb ? __ldg(rp + ra + lane) : 0, fe = ra + lane < rb ? __ldg(rp + ra + lane + 1) : 0;
        for (int q = ra; q < rb; q += 32) {
            const int r = q + lane;
            const int a = q == ra ? fs : r < rb ? __ldg(rp + r) : 0, b = q == ra ? fe : r < rb ? __ldg(rp + r + 1) : 0;
            if (b > a && b > tb && b <= te) B.end[b - 1 - tb] = 1;
        }
#pragma unroll
        for (int i = 0; i < 8; i++) B.vx[(32 * i + lane) / 8 * 9 + (lane & 7)] = make_double2(v[i], xv[i]);
        __syncwarp();
        load(t + nw);
        // the lane's entries; sums of rows that end go to their last entry's place
        const uint2 m = reinterpret_cast<const uint2 *>(B.end)[lane];
        double s = 0.0, f = 0.0;
        int first = -1;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            double2 &z = B.vx[lane * 9 + i];
            s = fma(z.x, z.y, s);
            if (((i < 4 ? m.x : m.y) >> 8 * (i & 3)) & 1u) {
                if (first < 0) {
                    first = i;
                    f = s;
                } else {
                    z.x = s;
                }
                s = 0.0;
            }
        }
        // the sums that lanes hand on: inclusive, back to the last lane in which a row ends
        bool stop = first >= 0;
        const bool any = __any_sync(0xffffffffu, stop);
        for (int o = 1; o < 32; o <<= 1) {
            const bool need = !stop && lane >= o;
            if (!__any_sync(0xffffffffu, need)) break;
            const double us = __shfl_up_sync(0xffffffffu, s, o);
            const bool ub = __shfl_up_sync(0xffffffffu, (int)stop, o);
            if (need) {
                s += us;
                stop = ub;
            }
        }
        const double in = __shfl_up_sync(0xffffffffu, s, 1);
        if (first >= 0) B.vx[lane * 9 + first].x = lane > 0 ? f + in : f;
        __syncwarp();
        for (int q = ra; q < rb; q += 32) {
            const int r = q + lane;
            const int a = q == ra ? fs : r < rb ? __ldg(rp + r) : 0, b = q == ra ? fe : r < rb ? __ldg(rp + r + 1) : 0;
            if (b > a && b > tb && b <= te) {
                const int e = b - 1 - tb;
                const double w = B.vx[e / 8 * 9 + (e & 7)].x;
                if (a < tb) D.tsum[t].x = w;
                else y[r] = beta == 0.0 ? alpha * w : fma(alpha, w, beta * y[r]);
            } else if (r < rb && a == b && beta == 0.0) {
                y[r] = 0.0;
            }
        }
        if (lane == 31) D.tsum[t].y = s;
        if (lane == 0) D.tinfo[t] = !any ? -1 : fs < tb ? ra : -2;
        __syncwarp();
    }
    __syncthreads();
    for (int q = t0 + threadIdx.x; q < t1; q += blockDim.x) {
        const int r = D.tinfo[q];
        if (r < 0) continue;
        double w = 0.0;
        for (int z = q - 1; z >= t0; z--) {
            w += D.tsum[z].y;
            if (D.tinfo[z] != -1) break;
        }
        w += D.tsum[q].x;
        y[r] = beta == 0.0 ? alpha * w : fma(alpha, w, beta * y[r]);
    }
}

__device__ void part_spmv(const xb_batch_dev &D, const Part &P, TileBuf *buf, int part, double alpha,
                          const double *x, double beta, double *y) {
    if (D.mode == 0) {
        const int *__restrict__ rp = D.rowptr;
        for (int r = P.r0 + threadIdx.x; r < P.r1; r += blockDim.x) {
            const double s = row_dot(D.col, D.val, x, __ldg(rp + r), __ldg(rp + r + 1));
            y[r] = beta == 0.0 ? alpha * s : fma(alpha, s, beta * y[r]);
        }
    } else {
        part_tiles(D, P, part, buf, alpha, x, beta, y);
    }
    // rows were stored by other threads than the ones that read them next,
    // so the CTA meets before anyone reads y
    __syncthreads();
}

// One block Gram-Schmidt pass over rows [r0, r1): w -= sum_{q < nu} c[q] V_{u0+q}
// (nu <= 4), then the nd <= 4 dots (w, V_{d0+q}) into a[] or, with NORM, (w, w)
// into a[0] and the nd <= 3 dots into a[1..].  Two rows per thread, every load
// of both issued before their arithmetic (the pass is latency-bound on one SM).
template <int R, bool NORM>
__device__ __forceinline__ void bgs_row(double *__restrict__ w, const double *__restrict__ V,
                                        int64_t ld, int u0, int nu, const double (&c)[4], int d0,
                                        int nd, int e0, int B, double (&a)[4]) {
    double x[R], pu[R][4], pd[R][4];
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int e = e0 + r * B;
        x[r] = w[e];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            pu[r][q] = q < nu ? V[(size_t)(u0 + q) * ld + e] : 0.0;
            pd[r][q] = q < nd ? V[(size_t)(d0 + q) * ld + e] : 0.0;
        }
    }
#pragma unroll
    for (int r = 0; r < R; r++) {
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (q < nu) x[r] = fma(-c[q], pu[r][q], x[r]);
        if (nu > 0) w[e0 + r * B] = x[r];
        if (NORM) a[0] = fma(x[r], x[r], a[0]);
#pragma unroll
        for (int q = 0; q < (NORM ? 3 : 4); q++)
            if (q < nd) a[NORM ? q + 1 : q] = fma(x[r], pd[r][q], a[NORM ? q + 1 : q]);
    }
}

template <bool NORM>
__device__ __forceinline__ void bgs_rows(double *__restrict__ w, const double *__restrict__ V,
                                         int64_t ld, int u0, int nu, const double (&c)[4], int d0,
                                         int nd, int r0, int r1, double (&a)[4]) {
#pragma unroll
    for (int q = 0; q < 4; q++) a[q] = 0.0;
    const int B = blockDim.x;
    int e = r0 + threadIdx.x;
    for (; e + B < r1; e += 2 * B) bgs_row<2, NORM>(w, V, ld, u0, nu, c, d0, nd, e, B, a);
    if (e < r1) bgs_row<1, NORM>(w, V, ld, u0, nu, c, d0, nd, e, B, a);
}

// MGS a vector at a time over rows [r0, r1): OP 0 returns (w, vn); OP 1 applies
// w -= c vp and returns (w, vn); OP 2 applies w -= c vp and returns (w, w).  Four
// rows per thread in flight.
template <int OP>
__device__ __forceinline__ double mgs_rows(double *__restrict__ w, const double *__restrict__ vp,
                                           const double *__restrict__ vn, double c, int r0, int r1) {
    const int B = blockDim.x;
    double a0 = 0.0, a1 = 0.0;
    auto row = [&](int e, double x, double p, double q, double &a) {
        if (OP != 0) {
            x = fma(-c, p, x);
            w[e] = x;
        }
        a = fma(x, OP == 2 ? x : q, a);
    };
    int e = r0 + threadIdx.x;
    for (; e + 3 * B < r1; e += 4 * B) {
        double x[4], p[4], q[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            x[u] = w[e + u * B];
            p[u] = OP != 0 ? vp[e + u * B] : 0.0;
            q[u] = OP != 2 ? vn[e + u * B] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 4; u++) row(e + u * B, x[u], p[u], q[u], u & 1 ? a1 : a0);
    }
    for (; e < r1; e += B) row(e, w[e], OP != 0 ? vp[e] : 0.0, OP != 2 ? vn[e] : 0.0, a0);
    return a0 + a1;
}

__device__ void solve_one(const xb_batch_dev &D, Part &P, Smem &S, TileBuf *buf, double tol, int maxiter,
                          unsigned long long deadline, int rank, double theta, int bcgs,
                          xb_batch_info *out) {
    const unsigned long long ts = gtimer();
    const int m_max = D.m_max;
    const int64_t ld = D.ld;
    double *V = D.V;
    double *H = D.H + (P.coop ? (size_t)rank * (m_max + 1) * m_max : 0);
    const int r0 = P.r0, r1 = P.r1;
    if (D.zero_x)
        for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) D.x[i] = 0.0;
    double a = 0.0;
    for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) a = fma(D.b[i], D.b[i], a);
    const double bnorm = sqrt(coop_sum(a, S, P));
    int iters = 0, restarts = 0, status = XB_OK, claimed = 0, m = D.m, K = 0;
    double tau = tol, res_true = 0.0;
    double samp[5];  // restart residuals for the MM-ratio rule (same in every thread)
    if (bnorm == 0.0) {
        for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) D.x[i] = 0.0;
    } else {
        for (;;) {
            coop_barrier(P);  // x complete before A x
            for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) V[i] = D.b[i];
            __syncthreads();  // the SpMV reads V_0 rows through other threads
            part_spmv(D, P, buf, rank, -1.0, D.x, 1.0, V);
            a = 0.0;
            for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) a = fma(V[i], V[i], a);
            const double beta = sqrt(coop_sum(a, S, P));
            // the time budget is rank 0's decision, broadcast by a reduction
            const double late =
                coop_sum((rank == 0 && threadIdx.x == 0 && gtimer() > deadline) ? 1.0 : 0.0, S, P);
            res_true = beta / bnorm;
            if (res_true <= tol) {
                status = XB_OK;
                break;
            }
            if (iters >= maxiter || late > 0.0) {
                status = XB_ENOCONV;
                break;
            }
            if (claimed) tau *= tol / res_true;  // fault convergence: narrow the threshold
            claimed = 0;
            if (restarts > 0) {  // restart-frequency rule (Eq. 1): judge every 5 samples
                samp[K++] = res_true;
                if (K == 5) {
                    double mx = samp[0], mn = samp[0];
                    for (int z = 1; z < 5; z++) {
                        mx = fmax(mx, samp[z]);
                        mn = fmin(mn, samp[z]);
                    }
                    if (mn > 0.0 && mx / mn < theta) m = min(m + 5, m_max);
                    K = 0;
                }
            }
            // the basis is stored unnormalised: v_i = sc_i V_i
            if (threadIdx.x == 0) {
                S.hn[0] = beta;
                S.sc[0] = 1.0 / beta;
            }
            __syncthreads();
            double gj = beta;  // warp 0: entry j of the least-squares right-hand side
            const double tol_g = tau * bnorm;
            const int lane = threadIdx.x & 31;
            int k = 0;
            for (int j = 0; j < m; j++) {
                iters++;
                double *w = V + (size_t)(j + 1) * ld;
                // v_j is complete: the norm's sum (or the residual's) ordered it
                part_spmv(D, P, buf, rank, S.sc[j], V + (size_t)j * ld, 0.0, w);
                // warp 2 keeps tt, the column's newest entry rotated by the earlier
                // rotations, and the sum of squares, a block behind
                double tt = 0.0, len2 = 0.0;
                int u0 = 0, nu = 0;
                auto take = [&]() {
                    for (int q = 0; q < nu; q++) {
                        const double h = S.hc[u0 + q];
                        len2 = fma(h, h, len2);
                        tt = u0 + q == 0 ? h : fma(-S.sn[u0 + q - 1], tt, S.cs[u0 + q - 1] * h);
                    }
                };
                // blocks of 4: one pass and one exchange each.  The dots of a block
                // are taken with the same w; for MGS they are corrected by the
                // block's own inner products: (w - sum_{k<i} c_k V_k, V_i) =
                // (w, V_i) - sum_{k<i} c_k (V_k, V_i), the same method with a quarter
                // of the exchanges.  Or (single_dots) MGS a vector at a time
                double c[4] = {0.0, 0.0, 0.0, 0.0}, a4[4];
                if (D.single) {
                    double ci = 0.0;
                    for (int i = 0; i <= j; i++) {
                        const double *vi = V + (size_t)i * ld;
                        double a1[1];
                        if (i == 0) a1[0] = mgs_rows<0>(w, nullptr, vi, 0.0, r0, r1);
                        else a1[0] = mgs_rows<1>(w, vi - ld, vi, ci, r0, r1);
                        const int ph = P.phase;
                        sums<1>(a1, S, P, take, [&](double &t) {
                            const double sq = S.sc[i];
                            t = (t * sq) * sq;
                            if (lane == 0) S.hc[i] = t * S.hn[i];
                        });
                        ci = S.tot[ph][0];
                        u0 = i;
                        nu = 1;
                    }
                    c[0] = ci;
                }
                for (int d0 = D.single ? j + 1 : 0; d0 <= j; d0 += 4) {
                    const int nd = min(4, j + 1 - d0);
                    bgs_rows<false>(w, V, ld, u0, nu, c, d0, nd, r0, r1, a4);
                    const int ph = P.phase;
                    sums<4>(a4, S, P, take, [&](double &t) {
                        const int q = lane >> 3;
                        const bool in = q < nd;
                        const double sq = in ? S.sc[d0 + q] : 0.0;
                        t = (t * sq) * sq;
                        if (!bcgs) {
#pragma unroll
                            for (int i = 0; i < 3; i++) {
                                const double ci = __shfl_sync(0xffffffffu, t, 8 * i);
                                if (in && q > i) t = fma(-ci, S.sg[(d0 + q) * 4 + i], t);
                            }
                        }
                        if (in && (lane & 7) == 0) S.hc[d0 + q] = t * S.hn[d0 + q];
                    });
#pragma unroll
                    for (int q = 0; q < 4; q++) c[q] = S.tot[ph][q];
                    u0 = d0;
                    nu = nd;
                }
                // the last projection, ||w||^2 and, for MGS, w's products with the
                // basis vectors it will share a block with
                const int ng = bcgs || D.single || j + 1 >= m ? 0 : (j + 1) & 3, g0 = j + 1 - ng;
                if (D.single) {
                    a4[0] = mgs_rows<2>(w, V + (size_t)j * ld, nullptr, c[0], r0, r1);
                    a4[1] = a4[2] = a4[3] = 0.0;
                } else {
                    bgs_rows<true>(w, V, ld, u0, nu, c, g0, ng, r0, r1, a4);
                }
                sums<4>(a4, S, P,
                        [&]() {
                            take();
                            if (lane == 0) {
                                S.tt = tt;
                                S.len2 = len2;
                            }
                            double *col = H + (size_t)j * (m_max + 1);
                            for (int i = lane; i <= j; i += 32) col[i] = S.hc[i];
                        },
                        [&](double &) {});
                // the new rotation (warp 0): both reciprocal roots in one sequence;
                // hypot where the square leaves the range in which it is exact enough
                if (threadIdx.x < 32) {
                    const double *tot = S.tot[P.phase ^ 1];
                    const double t0 = S.tt, hn2 = tot[0], rr2 = fma(t0, t0, hn2);
                    const double root = rsqrt(lane == 0 ? hn2 : rr2);
                    const double ihn = hn2 > 0.0 ? __shfl_sync(0xffffffffu, root, 0) : 0.0;
                    const double irr = __shfl_sync(0xffffffffu, root, 1);
                    const double hnj = hn2 * ihn;
                    double rr = rr2 * irr, c1 = t0 * irr, s1 = hnj * irr;
                    if (!(rr2 > 1e-280 && rr2 < 1e300)) {
                        rr = hypot(t0, hnj);
                        c1 = t0 / rr;
                        s1 = hnj / rr;
                    }
                    int flag = 0;
                    if (rr == 0.0) {
                        flag = 2;
                    } else {
                        if (lane == 0) {
                            S.cs[j] = c1;
                            S.sn[j] = s1;
                            S.g[j] = c1 * gj;
                            H[(size_t)j * (m_max + 1) + j + 1] = rr;  // the diagonal, until the restart
                            S.hn[j + 1] = hnj;
                            S.sc[j + 1] = ihn;
                        }
                        if (lane < ng) S.sg[(j + 1) * 4 + lane] = (tot[1 + lane] * ihn) * ihn;
                        gj = -s1 * gj;
                        if (hn2 <= 1e-28 * (S.len2 + hn2)) flag = 1;  // hn <= 1e-14 |column|
                        else if (fabs(gj) <= tol_g) flag = 3;
                    }
                    if (lane == 0) S.flag = flag;
                }
                __syncthreads();
                const int flag = S.flag;
                if (flag == 2) {
                    k = j;
                    status = XB_EBREAKDOWN;
                    break;
                }
                k = j + 1;
                if (flag != 0) {
                    claimed = 1;
                    break;
                }
                if (iters >= maxiter) break;
            }
            if (status == XB_EBREAKDOWN) break;
            // R y = g by columns on warp 0 (lane c holds g_c and 1 / R_cc; every
            // cooperating CTA holds the same R and g), then x += sum y_i sc_i V_i
            if (threadIdx.x < 32) {
                constexpr int QM = (XB_BATCH_MAX_M + 31) / 32;
                const int ldh = m_max + 1;
                // lane c rotates column c's entries with G_0..G_{c-1} (the arithmetic
                // of the steps' running value) and moves its diagonal into place
#pragma unroll
                for (int q = 0; q < QM; q++) {
                    const int cc = lane + 32 * q;
                    if (cc < k) {
                        double *col = H + (size_t)cc * ldh;
                        double tr = col[0];
                        for (int i = 1; i <= cc; i++) {
                            const double hi = col[i], cg_ = S.cs[i - 1], sg_ = S.sn[i - 1];
                            col[i - 1] = fma(cg_, tr, sg_ * hi);
                            tr = fma(-sg_, tr, cg_ * hi);
                        }
                        col[cc] = col[cc + 1];
                    }
                }
                __syncwarp();
                double gl[QM], dl[QM], hv[QM];
#pragma unroll
                for (int q = 0; q < QM; q++) {
                    const int cc = lane + 32 * q;
                    gl[q] = cc < k ? S.g[cc] : 0.0;
                    dl[q] = cc < k ? 1.0 / H[(size_t)cc * ldh + cc] : 0.0;
                    hv[q] = k > 0 && cc < k - 1 ? H[(size_t)(k - 1) * ldh + cc] : 0.0;
                }
                for (int i = k - 1; i >= 0; i--) {
                    const int qi = i >> 5, li = i & 31;
                    double gs = gl[0], ds = dl[0];
#pragma unroll
                    for (int q = 1; q < QM; q++)
                        if (qi == q) {
                            gs = gl[q];
                            ds = dl[q];
                        }
                    const double yi = __shfl_sync(0xffffffffu, gs, li) * __shfl_sync(0xffffffffu, ds, li);
                    if (lane == 0) S.yv[i] = yi * S.sc[i];
#pragma unroll
                    for (int q = 0; q < QM; q++) {
                        const int cc = lane + 32 * q;
                        if (32 * q < i && cc < i) gl[q] = fma(-hv[q], yi, gl[q]);
                        hv[q] = cc < i - 1 ? H[(size_t)(i - 1) * ldh + cc] : 0.0;  // the next column
                    }
                }
            }
            __syncthreads();
            {
                const double *__restrict__ Vc = V;
                double *__restrict__ xo = D.x;
                const int B = blockDim.x;
                int e = r0 + threadIdx.x;
                for (; e + B < r1; e += 2 * B) {  // two rows per thread in flight
                    double s0 = 0.0, s1 = 0.0;
                    for (int i = 0; i < k; i++) {
                        const double yi = S.yv[i];
                        s0 = fma(yi, Vc[(size_t)i * ld + e], s0);
                        s1 = fma(yi, Vc[(size_t)i * ld + e + B], s1);
                    }
                    xo[e] += s0;
                    xo[e + B] += s1;
                }
                for (; e < r1; e += B) {
                    double s0 = 0.0;
                    for (int i = 0; i < k; i++) s0 = fma(S.yv[i], Vc[(size_t)i * ld + e], s0);
                    xo[e] += s0;
                }
            }
            restarts++;
        }
    }
    if (threadIdx.x == 0 && rank == 0) {
        xb_batch_info inf;
        inf.status = status;
        inf.iters = iters;
        inf.restarts = restarts;
        inf.m = m;
        inf.mode = D.mode;
        inf.res_true = res_true;
        inf.ms = (double)(gtimer() - ts) * 1e-6;
        *out = inf;
    }
    __syncthreads();
}

__global__ void __cluster_dims__(kCl, 1, 1) __launch_bounds__(kBT, 1)
    k_batch_gmres(const xb_batch_dev *__restrict__ sys, xb_batch_info *__restrict__ out,
                  const int *__restrict__ order, int count, int nbig, int nsmall_cl,
                  int *__restrict__ queue, double tol, int maxiter, unsigned long long budget_ns,
                  double theta, int bcgs) {
    __shared__ Smem S;
    extern __shared__ __align__(16) unsigned char dyn[];
    TileBuf *buf = reinterpret_cast<TileBuf *>(dyn);
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    if (threadIdx.x == 0) S.t_start = gtimer();
    // one deadline for the whole cluster: rank 0's start plus the budget
    cl.sync();
    const unsigned long long deadline = cl.map_shared_rank(&S, 0)->t_start + budget_ns;
    cl.sync();
    // phase 1: the systems a whole cluster solves (order[0, nbig), largest
    // first), one per pull of the cluster's leader; phase 2: the single-CTA
    // systems (order[nbig, count), largest first), every CTA pulling its next
    // system as soon as it is free (no cluster barrier and no distributed
    // shared memory inside phase 2, so the CTAs of a cluster run apart).  The
    // first nsmall_cl clusters start with phase 2, so the longest single-CTA
    // solves do not wait for the end of phase 1, and join phase 1 when the
    // single-CTA queue is empty (their last systems are the smallest, so the
    // regrouping barrier waits little); the others run phase 1, then phase 2.
    const bool small_first = (int)(blockIdx.x / kCl) < nsmall_cl;  // cluster-uniform
    auto phase1 = [&]() {
        for (;;) {
            if (rank == 0 && threadIdx.x == 0) S.q = atomicAdd(queue, 1);
            cl.sync();
            const int q = cl.map_shared_rank(&S, 0)->q;
            cl.sync();  // the leader may overwrite q only after every CTA has read it
            if (q >= nbig) return;  // cluster-uniform
            const xb_batch_dev D = sys[order[q]];
            const int per = (D.n + kCl - 1) / kCl;
            Part P{min(D.n, rank * per), min(D.n, (rank + 1) * per), 1, 0};
            solve_one(D, P, S, buf, tol, maxiter, deadline, rank, theta, bcgs, out + order[q]);
        }
    };
    auto phase2 = [&]() {
        for (;;) {
            if (threadIdx.x == 0) S.q = atomicAdd(queue + 1, 1);
            __syncthreads();
            const int q = nbig + S.q;
            __syncthreads();  // S.q is rewritten only after every thread has read it
            if (q >= count) return;  // CTA-uniform
            const xb_batch_dev D = sys[order[q]];
            Part P{0, D.n, 0, 0};
            solve_one(D, P, S, buf, tol, maxiter, deadline, 0, theta, bcgs, out + order[q]);
        }
    };
    if (small_first) {
        phase2();
        cl.sync();  // every CTA of the cluster is free: take cluster systems
        phase1();
    } else {
        phase1();
        phase2();
    }
}

constexpr int kDyn = (int)sizeof(TileBuf) * (kBT / 32);

// Mode 1's tiles of a system whose host row pointer is rp: tptr and, appended to
// trow, the tiles' rows.
void cut_tiles(xb_batch_dev &d, const int *rp, std::vector<int> &trow) {
    const int parts = d.coop ? kCl : 1, per = (d.n + parts - 1) / parts;
    const size_t base = trow.size();
    for (int c = 0; c < kCl; c++) {
        d.tptr[c] = (int)(trow.size() - base);
        if (c >= parts) continue;
        int r = std::min(d.n, c * per);
        const int r1 = std::min(d.n, (c + 1) * per);
        for (int64_t e = rp[r]; e < rp[r1]; e += kTile) {
            while (rp[r + 1] <= e) r++;
            trow.push_back(r);
        }
    }
    d.tptr[kCl] = (int)(trow.size() - base);
}

// Whole clusters of the kernel that fit on the GPU at once.
int resident_clusters(size_t dyn) {
    cudaLaunchConfig_t lc;
    std::memset(&lc, 0, sizeof lc);
    lc.gridDim = dim3(kCl, 1, 1);
    lc.blockDim = dim3(kBT, 1, 1);
    lc.dynamicSmemBytes = dyn;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, (void *)k_batch_gmres, &lc) != cudaSuccess || clusters < 1) {
        cudaGetLastError();
        clusters = xb::num_sms() / kCl;
    }
    return std::max(1, clusters);
}

// Estimated time of an Arnoldi step, in us, at the cycle's mean basis size m / 2:
// 2 + m / 8 sums at 2 us (3.3 us across a cluster), and n m + nnz FP64 terms (1.5
// nnz in mode 1) at 0.4 ns a CTA, with a seventh lost to the split over a cluster's
// 8.  Fitted to 48 systems of 1000 to 57,000 rows at m = 30 (one CTA 28 to 825 us,
// a cluster 18 to 133 us a step), within a fifth.  At m = 10 it is a third too low for
// both, at m = 100 a sixth too high; the split of five mixes of 20 to 300 systems is
// within 14% of the best fixed number of rows at m = 10, 30 and 100.
double step_us(const xb_batch_dev &d, bool cluster) {
    const double sums = 2.0 + d.m / 8.0,
                 terms = 4e-4 * ((double)d.m * d.n + (d.mode == 1 ? 1.5 : 1.0) * d.nnz);
    return cluster ? 3.3 * sums + 1.15 * terms / kCl : 2.0 * sums + terms;
}

// Whether MGS takes a system's basis a vector at a time, an exchange each, instead
// of in corrected blocks of 4.  A block saves exchanges (2 us, 3.3 across a
// cluster) but takes up to 3 more dots a step for its own products and has fewer
// rows of the vectors on their way, so it loses where a CTA has many rows for the
// cycle's length.  Us a step, blocks / singly, one CTA: n = 1600, m = 5, 10, 20:
// 24.2 / 20.9, 25.5 / 24.4, 31.5 / 34.1; n = 6400, m = 20, 30, 50: 91 / 84, 113 / 110,
// 153 / 161; n = 28,900, m = 10, 30, 100: 341 / 275, 481 / 433, 1044 / 1072.  A
// cluster: n = 40,000, m = 10, 20, 30: 61.5 / 54.1, 79.4 / 81.1, 98 / 108; n =
// 202,500, m = 5, 20, 60: 305 / 243, 359 / 318, 638 / 642.
int single_dots(const xb_batch_dev &d, int bcgs) {
    const double rows = d.coop ? (d.n + kCl - 1) / kCl : d.n;
    return !bcgs && rows >= (d.coop ? 2.4 : 1.5) * d.m * (d.m + 100.0);
}

// Decides which systems a whole cluster solves and returns the order of the
// queues: the cluster's systems first, each part largest first, so that the long
// solves start in the first wave.  A cluster solves a system sooner but at up to 8
// times the SM time.  From kLargeN rows on it takes a system always: step counts
// and row lengths are unknown, and a long solve on one CTA can outlast all others
// (512 systems, some of which run 3000 steps: 24.2 s without this, 15.0 with it).
// Of the others the k largest follow, for the k whose estimated end is first: no
// earlier than the longest cluster solve, than the longest single-CTA one, and than
// all the work spread over the resident CTAs, at equal step counts.  Few systems
// thus all go to clusters, many small ones to a CTA each.  The environment variable
// XB_BATCH_COOP_MIN_N sets the number of rows and leaves the estimate out.
std::vector<int> split_systems(std::vector<xb_batch_dev> &h, int clusters) {
    const int count = (int)h.size();
    const char *env = std::getenv("XB_BATCH_COOP_MIN_N");
    const long coop_min = env ? std::max(1L, std::atol(env)) : kLargeN;
    for (xb_batch_dev &d : h) d.coop = d.n >= coop_min ? 1 : 0;
    std::vector<int> order(count);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        if (h[a].coop != h[b].coop) return h[a].coop > h[b].coop;
        return step_us(h[a], false) > step_us(h[b], false);
    });
    if (env) return order;
    double spread = 0.0;  // SM time of all systems with the first k in clusters
    double best = 0.0, longest = 0.0;
    int first = 0, take = 0;
    for (const xb_batch_dev &d : h) {
        const double c = step_us(d, true);
        spread += d.coop ? kCl * c : step_us(d, false);
        if (d.coop) longest = std::max(longest, c);
        first += d.coop;
    }
    for (int k = first; k <= count; k++) {
        const double alone = k < count ? step_us(h[order[k]], false) : 0.0;
        const double end = std::max({longest, alone, spread / (kCl * clusters)});
        if (k == first || end <= best) {  // a tie: the shorter solves
            best = end;
            take = k;
        }
        if (k == count) break;
        const double c = step_us(h[order[k]], true);
        longest = std::max(longest, c);
        spread += kCl * c - alone;
    }
    for (int k = first; k < take; k++) h[order[k]].coop = 1;
    return order;
}

}  // namespace

namespace xb {

// One system through the persistent kernel: a single 8-CTA cluster solving
// it together (rows split over the 8 CTAs, dot products combined through
// distributed shared memory), the system's basis and Hessenberg, its
// descriptor, queue and result in the plan's workspace; no graph capture, no
// allocation after the workspace has grown.  Used by gmres_solve for small
// systems, whose multi-launch Arnoldi steps are bound by launch and
// synchronisation latency.  The whole cluster is used even below the batch's
// cluster threshold: the launch holds one cluster anyway, and 8 SMs hide more
// of the L2 latency of each Gram-Schmidt pass (n = 4096: 12.2 ms for 535 steps).
int batch_single(xb_plan *p, const double *b, double *x, const xb_options &o, int mode,
                 xb_info &inf, double *alg_bytes, cudaStream_t s) {
    xb_batch_dev d;
    std::memset(&d, 0, sizeof d);
    d.n = p->n;
    d.nnz = p->nnz;
    d.m = o.m;
    d.m_max = o.dafrt ? std::max(o.m, std::min(o.m_max, XB_BATCH_MAX_M)) : o.m;
    d.mode = mode;
    d.zero_x = 0;
    d.coop = 1;
    d.ld = ((int64_t)d.n + 31) / 32 * 32;
    d.rowptr = p->rowptr;
    d.col = p->col;
    d.val = p->val;
    d.b = b;
    d.x = x;
    const int bcgs = o.ortho == XB_ORTHO_BCGS ? 1 : 0;
    d.single = single_dots(d, bcgs);
    const size_t nv = (size_t)(d.m_max + 1) * d.ld;
    const size_t nh = (size_t)(d.coop ? kCl : 1) * (d.m_max + 1) * d.m_max + 32;
    const size_t meta = 4096;  // descriptor, result, order, queue
    // mode 1: the tiles, from the plan's host row pointer
    std::vector<int> trow;
    std::memset(d.tptr, 0, sizeof d.tptr);
    if (mode == 1) {
        std::vector<int> rp_h;
        const int *rp = p->h_rowptr.data();
        if ((int)p->h_rowptr.size() != p->n + 1) {
            rp_h.resize((size_t)p->n + 1);
            XB_CUDA(cudaMemcpyAsync(rp_h.data(), p->rowptr, rp_h.size() * sizeof(int), cudaMemcpyDeviceToHost, s));
            XB_CUDA(cudaStreamSynchronize(s));
            rp = rp_h.data();
        }
        cut_tiles(d, rp, trow);
    }
    const size_t nt = trow.size();
    XB_TRY(ensure_work(p, (nv + nh) * sizeof(double) + meta + nt * (sizeof(double2) + 2 * sizeof(int))));
    char *w = static_cast<char *>(p->d_work);
    d.V = reinterpret_cast<double *>(w);
    d.H = d.V + nv;
    char *m0 = w + (nv + nh) * sizeof(double);
    xb_batch_dev *d_sys = reinterpret_cast<xb_batch_dev *>(m0);
    xb_batch_info *d_info = reinterpret_cast<xb_batch_info *>(m0 + 1024);
    int *d_order = reinterpret_cast<int *>(m0 + 2048);
    int *d_queue = d_order + 1;
    static_assert(sizeof(xb_batch_dev) <= 1024 && sizeof(xb_batch_info) <= 1024, "meta layout");
    d.tsum = reinterpret_cast<double2 *>(m0 + meta);
    d.tinfo = reinterpret_cast<int *>(d.tsum + nt);
    d.trow = d.tinfo + nt;
    if (nt > 0)
        XB_CUDA(cudaMemcpyAsync(d.tinfo + nt, trow.data(), nt * sizeof(int), cudaMemcpyHostToDevice, s));
    const int zero = 0;
    XB_CUDA(cudaMemcpyAsync(d_sys, &d, sizeof d, cudaMemcpyHostToDevice, s));
    XB_CUDA(cudaMemcpyAsync(d_order, &zero, sizeof zero, cudaMemcpyHostToDevice, s));
    XB_CUDA(cudaMemsetAsync(d_queue, 0, 2 * sizeof(int), s));
    const unsigned long long budget = (unsigned long long)(std::min(o.maxtime_s, 3600.0) * 1e9);
    const double theta = o.dafrt ? o.dafrt_theta : 0.0;
    XB_CUDA(cudaFuncSetAttribute(k_batch_gmres, cudaFuncAttributeMaxDynamicSharedMemorySize, kDyn));
    k_batch_gmres<<<kCl, kBT, mode == 1 ? kDyn : 0, s>>>(d_sys, d_info, d_order, 1, 1, 0, d_queue, o.tol, o.maxiter,
                                      budget, theta, bcgs);
    XB_LAUNCHED("k_batch_gmres (single system)");
    xb_batch_info r;
    XB_CUDA(cudaMemcpyAsync(&r, d_info, sizeof r, cudaMemcpyDeviceToHost, s));
    XB_CUDA(cudaStreamSynchronize(s));
    inf.iters = r.iters;
    inf.restarts = r.restarts;
    inf.m_final = r.m;
    inf.res_true = r.res_true;
    inf.ortho_used = bcgs ? XB_ORTHO_BCGS : XB_ORTHO_MGS;
    inf.persistent = 1;
    // algorithmic bytes: per Arnoldi step one SpMV and the Gram-Schmidt passes
    // at the cycle's mean basis size, plus a residual per restart
    const double jm = (r.m + 1) / 2.0, n = d.n;
    *alg_bytes = r.iters * (spmv_alg_bytes(p, false, 8) + (2.0 * jm + 2.0) * 8.0 * n) +
                 (r.restarts + 1) * (spmv_alg_bytes(p, true, 8) + 16.0 * n);
    if (r.status == XB_ENOCONV)
        return set_error(XB_ENOCONV, "not converged: ||b-Ax||/||b|| = %.3e > tol %.1e", r.res_true,
                         o.tol);
    return r.status;
}

}  // namespace xb

extern "C" {

int xb_batch_destroy(xb_batch *bt) {
    if (!bt) return XB_OK;
    cudaDeviceSynchronize();
    if (bt->exec) cudaGraphExecDestroy(bt->exec);
    if (bt->graph) cudaGraphDestroy(bt->graph);
    cudaFree(bt->d_sys);
    cudaFree(bt->d_info);
    cudaFree(bt->d_order);
    cudaFree(bt->d_queue);
    cudaFree(bt->d_ws);
    cudaFree(bt->d_tiles);
    delete bt;
    return XB_OK;
}

int xb_batch_create(int32_t count, const xb_batch_sys *sys, const xb_options *opt, void *stream,
                    xb_batch **out) {
    if (count < 0 || (count > 0 && !sys) || !out) return xb::set_error(XB_EINVAL, "batch_create: bad argument");
    *out = nullptr;
    // the systems' arrays may still be on their way on the caller's stream, which
    // the legacy default stream does not wait for
    cudaStream_t s = (cudaStream_t)stream;
    xb_options o;
    if (opt) o = *opt;
    else xb_options_default(&o);
    if (!(o.tol > 0.0)) return xb::set_error(XB_EINVAL, "batch_create: tol must be > 0");
    if (o.ortho != XB_ORTHO_MGS && o.ortho != XB_ORTHO_BCGS && o.ortho != XB_ORTHO_AUTO)
        return xb::set_error(XB_EINVAL, "batch_create: orthogonalisation must be MGS, BCGS or AUTO");
    std::vector<xb_batch_dev> h(count);
    size_t ws = 0;
    for (int i = 0; i < count; i++) {
        const xb_batch_sys &q = sys[i];
        if (q.n < 0 || q.nnz < 0 || q.m < 1 || q.m > XB_BATCH_MAX_M || (q.mode != 0 && q.mode != 1) ||
            (q.n > 0 && (!q.rowptr || !q.b || !q.x || (q.nnz > 0 && (!q.col || !q.val)))))
            return xb::set_error(XB_EINVAL, "batch_create: system %d invalid (n=%d m=%d mode=%d)", i,
                                 q.n, q.m, q.mode);
        xb_batch_dev &d = h[i];
        d.n = q.n;
        d.nnz = q.nnz;
        d.m = q.m;
        d.m_max = o.dafrt ? std::max(q.m, std::min(o.m_max, XB_BATCH_MAX_M)) : q.m;
        d.mode = q.mode;
        d.zero_x = q.zero_x;
        d.ld = ((int64_t)q.n + 31) / 32 * 32;
        d.rowptr = q.rowptr;
        d.col = q.col;
        d.val = q.val;
        d.b = q.b;
        d.x = q.x;
    }
    cudaError_t e = cudaFuncSetAttribute(k_batch_gmres, cudaFuncAttributeMaxDynamicSharedMemorySize, kDyn);
    if (e != cudaSuccess) return xb::cuda_error(e, "batch_create: shared memory");
    // without mode 1 its tiles' shared memory is left to the L1
    const size_t dyn = std::any_of(h.begin(), h.end(), [](const xb_batch_dev &d) { return d.mode == 1; }) ? kDyn : 0;
    const int clusters = resident_clusters(dyn);
    const std::vector<int> order = split_systems(h, clusters);
    for (const xb_batch_dev &d : h)
        ws += (size_t)(d.m_max + 1) * d.ld + (size_t)(d.coop ? kCl : 1) * (d.m_max + 1) * d.m_max + 32;
    // mode 1: each system's tiles, from a host copy of its row pointer
    std::vector<int> trow, rp_h;
    std::vector<size_t> toff(count, 0);
    for (int i = 0; i < count; i++) {
        std::memset(h[i].tptr, 0, sizeof h[i].tptr);
        h[i].trow = nullptr;
        h[i].tinfo = nullptr;
        h[i].tsum = nullptr;
        toff[i] = trow.size();
        if (h[i].mode != 1 || h[i].n < 1 || h[i].nnz < 1) continue;
        rp_h.resize((size_t)h[i].n + 1);
        e = cudaMemcpyAsync(rp_h.data(), h[i].rowptr, rp_h.size() * sizeof(int), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return xb::cuda_error(e, "batch_create: read rowptr");
        cut_tiles(h[i], rp_h.data(), trow);
    }
    xb_batch *bt = new xb_batch();
    bt->count = count;
    auto fail = [&](int code) {
        xb_batch_destroy(bt);
        return code;
    };
    e = cudaMalloc(&bt->d_ws, std::max<size_t>(ws, 1) * sizeof(double));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(xb::set_error(XB_ENOMEM, "batch_create: %zu bytes of workspace", ws * 8));
    }
    const size_t nt = trow.size();
    if (nt > 0) {
        e = cudaMalloc(&bt->d_tiles, nt * (sizeof(double2) + 2 * sizeof(int)));
        if (e != cudaSuccess) {
            cudaGetLastError();
            return fail(xb::set_error(XB_ENOMEM, "batch_create: tiles"));
        }
        double2 *ts = static_cast<double2 *>(bt->d_tiles);
        int *ti = reinterpret_cast<int *>(ts + nt);
        e = cudaMemcpyAsync(ti + nt, trow.data(), nt * sizeof(int), cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) return fail(xb::cuda_error(e, "batch_create: tiles"));
        for (int i = 0; i < count; i++) {
            h[i].tsum = ts + toff[i];
            h[i].tinfo = ti + toff[i];
            h[i].trow = ti + nt + toff[i];
        }
    }
    // orthogonalisation: MGS or BCGS (block length 4); the accuracy policy's
    // choice for AUTO (no fault switch inside the launch)
    const int ortho = o.ortho == XB_ORTHO_AUTO ? (o.tol <= 1e-10 ? XB_ORTHO_MGS : XB_ORTHO_BCGS)
                                               : o.ortho;
    const int bcgs = ortho == XB_ORTHO_BCGS ? 1 : 0;
    size_t off = 0;
    for (int i = 0; i < count; i++) {
        h[i].single = single_dots(h[i], bcgs);
        h[i].V = bt->d_ws + off;
        off += (size_t)(h[i].m_max + 1) * h[i].ld;
        h[i].H = bt->d_ws + off;
        off += (size_t)(h[i].coop ? kCl : 1) * (h[i].m_max + 1) * h[i].m_max + 32;
    }
    int nbig = 0;
    for (int i = 0; i < count; i++) nbig += h[i].coop ? 1 : 0;
    e = cudaMalloc(&bt->d_sys, std::max(count, 1) * sizeof(xb_batch_dev));
    if (e == cudaSuccess) e = cudaMalloc(&bt->d_info, std::max(count, 1) * sizeof(xb_batch_info));
    if (e == cudaSuccess) e = cudaMalloc(&bt->d_order, std::max(count, 1) * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&bt->d_queue, 2 * sizeof(int));
    if (e == cudaSuccess && count > 0)
        e = cudaMemcpyAsync(bt->d_sys, h.data(), count * sizeof(xb_batch_dev), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && count > 0)
        e = cudaMemcpyAsync(bt->d_order, order.data(), count * sizeof(int), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // a run may be on another stream
    if (e != cudaSuccess) return fail(xb::cuda_error(e, "batch_create"));
    bt->grid = kCl * clusters;  // persistent: as many whole clusters as can be co-resident
    // clusters that take the single-CTA systems from the start: their share
    // of the work; none without cluster systems to balance against
    double w_big = 0.0, w_small = 0.0;
    for (const xb_batch_dev &d : h) (d.coop ? w_big : w_small) += d.coop ? kCl * step_us(d, true) : step_us(d, false);
    int nsmall_cl = 0;
    if (nbig > 0 && w_small > 0.0)
        nsmall_cl = std::min(clusters - 1, (int)std::lround(clusters * w_small / (w_big + w_small)));
    const unsigned long long budget = (unsigned long long)(std::min(o.maxtime_s, 3600.0) * 1e9);
    const double theta = o.dafrt ? o.dafrt_theta : 0.0;  // theta 0: the rule never fires
    // capture on a private stream (the caller's may be the legacy default
    // stream, which cannot be captured): reset the queue, one persistent launch
    cudaStream_t cs = nullptr;
    e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) return fail(xb::cuda_error(e, "batch_create: capture stream"));
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) {
        cudaStreamDestroy(cs);
        return fail(xb::cuda_error(e, "batch_create: begin capture"));
    }
    cudaMemsetAsync(bt->d_queue, 0, 2 * sizeof(int), cs);
    k_batch_gmres<<<bt->grid, kBT, dyn, cs>>>(bt->d_sys, bt->d_info, bt->d_order, count, nbig,
                                             nsmall_cl, bt->d_queue,
                                             o.tol, o.maxiter, budget, theta, bcgs);
    cudaError_t el = cudaGetLastError();
    e = cudaStreamEndCapture(cs, &bt->graph);
    cudaStreamDestroy(cs);
    if (el != cudaSuccess) return fail(xb::cuda_error(el, "batch_create: launch in capture"));
    if (e != cudaSuccess) return fail(xb::cuda_error(e, "batch_create: end capture"));
    e = cudaGraphInstantiate(&bt->exec, bt->graph, 0);
    if (e != cudaSuccess) return fail(xb::cuda_error(e, "batch_create: instantiate"));
    *out = bt;
    return XB_OK;
}

int xb_batch_run(xb_batch *bt, void *stream) {
    if (!bt) return xb::set_error(XB_EINVAL, "batch_run: NULL");
    if (bt->count == 0) return XB_OK;
    XB_CUDA(cudaGraphLaunch(bt->exec, (cudaStream_t)stream));
    return XB_OK;
}

int xb_batch_results(xb_batch *bt, xb_batch_info *infos, void *stream) {
    if (!bt || (bt->count > 0 && !infos)) return xb::set_error(XB_EINVAL, "batch_results: bad argument");
    if (bt->count == 0) return XB_OK;
    cudaStream_t s = (cudaStream_t)stream;
    XB_CUDA(cudaMemcpyAsync(infos, bt->d_info, bt->count * sizeof(xb_batch_info), cudaMemcpyDeviceToHost, s));
    XB_CUDA(cudaStreamSynchronize(s));
    int worst = XB_OK;
    for (int i = 0; i < bt->count; i++)
        if (infos[i].status != XB_OK && worst == XB_OK) worst = infos[i].status;
    return worst;
}

int xb_batch_solve(int32_t count, const xb_batch_sys *sys, const xb_options *opt,
                   xb_batch_info *infos, void *stream) {
    xb_batch *bt = nullptr;
    XB_TRY(xb_batch_create(count, sys, opt, stream, &bt));
    int r = xb_batch_run(bt, stream);
    if (r == XB_OK) r = xb_batch_results(bt, infos, stream);
    xb_batch_destroy(bt);
    return r;
}

}  // extern "C"
