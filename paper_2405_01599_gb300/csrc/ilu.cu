// ILU(0) preconditioner (the preconditioner of the paper's solver runs,
// Sec. 4.3): incomplete LU factorization in the sparsity pattern of A
// (general CRS), applied as z = U^{-1} L^{-1} r.
//
// Setup: the host derives, from the pattern alone, the dependency level of
// every row for the forward substitution (level(i) = 1 + max level(k) over the
// stored k < i in row i) and for the backward one (over the stored j > i).  The
// numeric factorization runs level by level on the device, one warp per row:
// for each stored (i, k), k < i, in ascending k, l_ik = a_ik / u_kk, and every
// stored (i, j), j > k, subtracts l_ik u_kj when (k, j) is stored (binary search
// in row k, which an earlier level finished).  Both substitutions run in one
// launch in which rows wait for the values they need (the flow path), or as one
// kernel per level and row tier, captured once in a CUDA graph (the graph path).
#include "common.cuh"

#include <algorithm>
#include <climits>
#include <cstdlib>
#include <cmath>
#include <thread>

namespace {

constexpr int kLongRow = 512;  // triangle entries above which a row gets a CTA
constexpr int kEllMax = 8;     // triangle entries up to which a row is stored as ELL

__device__ __forceinline__ int find_in_row(const int *__restrict__ ci, int lo, int hi, int j) {
    // search [lo, hi) of a sorted column list for j
    hi -= 1;
    while (lo <= hi) {
        const int mid = lo + ((hi - lo) >> 1);
        const int c = __ldg(ci + mid);
        if (c == j) return mid;
        if (c < j) lo = mid + 1;
        else hi = mid - 1;
    }
    return -1;
}

// Factor the rows listed in rows[0..cnt) (one dependency level), warp per row.
__global__ void k_ilu_factor(int cnt, const int *__restrict__ rows, const int *__restrict__ rp,
                             const int *__restrict__ ci, const int *__restrict__ dpos,
                             double *__restrict__ lu, int *__restrict__ flag) {
    const int lane = threadIdx.x & 31;
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= cnt) return;  // warp-uniform
    const int i = rows[w];
    const int a = rp[i], e = rp[i + 1], d = dpos[i];
    for (int p = a; p < d; p++) {
        const int k = __ldg(ci + p);
        const int dk = dpos[k];
        const double piv = lu[dk];
        if (piv == 0.0) {
            if (lane == 0) atomicExch(flag, 1);
            return;
        }
        const double lik = lu[p] / piv;
        __syncwarp();
        if (lane == 0) lu[p] = lik;
        const int ke = rp[k + 1];
        for (int q = p + 1 + lane; q < e; q += 32) {
            const int pos = find_in_row(ci, dk + 1, ke, __ldg(ci + q));
            if (pos >= 0) lu[q] = fma(-lik, lu[pos], lu[q]);
        }
        __syncwarp();  // row i's entries settled before the next l_ik is formed
    }
    if (lane == 0 && lu[d] == 0.0) atomicExch(flag, 1);
}

// One level of a substitution.  FWD: z_i = r_i - sum_{k<i} l_ik z_k over the
// stored strictly lower entries.  Backward: z_i = (z_i - sum_{j>i} u_ij z_j) / u_ii.
template <bool FWD>
__global__ void __launch_bounds__(256) k_ilu_level(int cnt, const int *__restrict__ rows,
                                                   const int *__restrict__ rp,
                                                   const int *__restrict__ ci,
                                                   const int *__restrict__ dpos,
                                                   const double *__restrict__ lu,
                                                   const double *__restrict__ r,
                                                   double *__restrict__ z) {
    const int lane = threadIdx.x & 31;
    const int base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31;  // warp's first slot
    if (base >= cnt) return;  // warp-uniform
    const int slot = base + lane;
    int i = -1, ka = 0, kb = 0;
    if (slot < cnt) {
        i = rows[slot];
        const int d = dpos[i];
        ka = FWD ? rp[i] : d + 1;
        kb = FWD ? d : rp[i + 1];
    }
    const bool lng = kb - ka > 32;
    double s = 0.0;
    if (!lng)
        for (int k = ka; k < kb; k++) s = fma(__ldg(lu + k), z[__ldg(ci + k)], s);
    unsigned todo = __ballot_sync(0xffffffffu, lng);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const int la = __shfl_sync(0xffffffffu, ka, src);
        const int lb = __shfl_sync(0xffffffffu, kb, src);
        double t = 0.0;
        for (int k = la + lane; k < lb; k += 32) t = fma(__ldg(lu + k), z[__ldg(ci + k)], t);
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == src) s = t;
    }
    if (i >= 0) {
        if (FWD) z[i] = r[i] - s;
        else z[i] = (z[i] - s) / lu[dpos[i]];
    }
}

// One level's long rows, a CTA per row (block reduction in a fixed order).
template <bool FWD>
__global__ void __launch_bounds__(256) k_ilu_level_long(const int *__restrict__ rows,
                                                        const int *__restrict__ rp,
                                                        const int *__restrict__ ci,
                                                        const int *__restrict__ dpos,
                                                        const double *__restrict__ lu,
                                                        const double *__restrict__ r,
                                                        double *__restrict__ z) {
    __shared__ double sh[8];
    const int i = rows[blockIdx.x];
    const int d = dpos[i];
    const int ka = FWD ? rp[i] : d + 1, kb = FWD ? d : rp[i + 1];
    double t = 0.0;
    for (int k = ka + threadIdx.x; k < kb; k += blockDim.x)
        t = fma(__ldg(lu + k), z[__ldg(ci + k)], t);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) s += sh[w];
        if (FWD) z[i] = r[i] - s;
        else z[i] = (z[i] - s) / lu[d];
    }
}

// One level's short rows in ELL form, a thread per row: the row index, its
// entries and (backward) its pivot are independent loads, then the gathers.
template <bool FWD>
__global__ void __launch_bounds__(256) k_ilu_ell(int cnt, int width, const int *__restrict__ rows,
                                                 const int *__restrict__ ecol,
                                                 const double *__restrict__ eval,
                                                 const double *__restrict__ diag,
                                                 const double *__restrict__ r,
                                                 double *__restrict__ z) {
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= cnt) return;
    const int i = __ldg(rows + slot);
    double s = 0.0;
    for (int t = 0; t < width; t++) {
        const long long e = (long long)t * cnt + slot;
        s = fma(__ldg(eval + e), z[__ldg(ecol + e)], s);
    }
    if (FWD) z[i] = r[i] - s;
    else z[i] = (z[i] - s) / __ldg(diag + slot);
}

// ELL values from the factors (padding entries stay 0), and the pivots in
// backward level order.
__global__ void k_ell_fill(long long cnt, const int *__restrict__ src,
                           const double *__restrict__ lu, double *__restrict__ val) {
    const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (e < cnt) val[e] = src[e] >= 0 ? lu[src[e]] : 0.0;
}
__global__ void k_diag_fill(int n, const int *__restrict__ rows, const int *__restrict__ dpos,
                            const double *__restrict__ lu, double *__restrict__ diag,
                            double *__restrict__ rdiag, int *__restrict__ odd) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const double d = lu[dpos[rows[s]]];
    diag[s] = d;
    if (rdiag) {
        rdiag[s] = 1.0 / d;
        if (!(fabs(d) > 1e-280 && fabs(d) < 1e280)) *odd = 1;  // d and 1 / d in the normal range?
    }
}

// ---- flow substitution ---------------------------------------------------------
// Both substitutions in one cooperative launch without barriers between
// levels.  CTA c owns a block of consecutive rows, in both triangles, and takes
// its rows in level order as items: up to 32 rows of one level (a lane each),
// or fewer rows with 2 to 32 lanes each, so that no lane has more than four
// entries, or one longer row (the warp).  A row's value is published as soon as it is
// formed and a row waits for the very values it needs: those of the CTA's own
// rows in shared memory, the others in device memory, where a value travels as
// two 8-byte words that both carry the number of the application (so nothing
// is reset between applications and no fence is needed).
//
// What bounds it: the longest chain of rows, one hop per level.  A hop through
// shared memory takes 0.4 us (an FP64 FMA alone 0.1), one through device memory
// 1.0 us and, with every CTA waiting on others, up to 2; the level barrier this
// replaces took ~6 us and a kernel per level ~4 us.  Consecutive rows per CTA
// keep most hops of a stencil inside a CTA.  One application (GB300; the graph
// of level launches or the level barrier, whichever was faster, in brackets):
// 96^3 convection-diffusion 0.62-0.65 ms (2.0), 64^3 0.26, 30^3 0.11 (0.44), 180^3
// (blocks too large for shared memory) 2.6 (4.3), power-law rows n = 20,000 0.09
// (1.1), n = 1M 0.50 (3.4).
//
// Four entries a lane: an item is one round of loads and waits.  With a lane for
// a row of up to 32 entries (up to 5 rounds of ~2 us, and the rows of a power law's
// late levels are long) n = 1M took 1.04 ms, n = 20,000 0.46 and 0.16 with four (2048
// rows a block); with 2 / 3 / 6 entries a lane 0.76 / 0.54 / 0.49 and 0.23 / 0.18 / 0.19.  The lanes'
// sums meet in a tree: against exact arithmetic 4.5e-17 of ||z||, one by one 4.6e-17
// (power law, n = 200,000).
//
// Every wait ends: warps take a CTA's items in level order, so of the rows not
// yet done in the whole grid those of the lowest level wait for nothing; and a
// wait is bounded all the same (`polls` polls, or `limit` ns): then the kernel
// sets the error flag and every warp leaves at its next poll.
constexpr int kFlowWarps = 16;
constexpr int kFlowFirst = 4;    // entries of each kind a lane has: all on their way at once
constexpr int kFlowGroup = 8;    // entries a lane loads together in such a row
constexpr unsigned long long kNotReady = 0xffffffffffffffffull;  // a NaN that is never stored

struct FlowTri {
    const int4 *items;      // {first slot, rows | long << 8 | log2(lanes of a row) << 9,
                            //  a lane's remote | local entries << 16, entries from ebase}
    const int *iptr;        // per CTA: its items
    const long long *ebase; // per CTA: its entries
    const int *rows;        // slot -> row
    const int *ecol;        // remote: column; local: row of the block; -1: none
    const double *eval;
    const double *diag, *rdiag;  // by slot (backward): pivot and its reciprocal
};
struct FlowArgs {
    FlowTri L, U;
    const int *bstart;      // per CTA: first row
    const int *rp, *ci, *dpos;
    const double *lu, *r;
    double *z;
    ulonglong2 *ty, *tz;    // published values of the two substitutions
    unsigned seq, polls, look;  // polls of one wait (0: the clock decides); polls between looks
    unsigned long long limit;
    volatile int *err;      // host-visible
    int *stop;              // the same for the grid
    int cap;                // rows whose values shared memory holds
};

__device__ __forceinline__ void flow_put(ulonglong2 *p, double v, unsigned seq) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned long long s = (unsigned long long)seq << 32;
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(s | (b & 0xffffffffu)),
                 "l"(s | (b >> 32)) : "memory");
}
__device__ __forceinline__ bool flow_get(const ulonglong2 *p, unsigned seq, double &v) {
    unsigned long long x, y;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
    v = __longlong_as_double((long long)((x & 0xffffffffu) | (y << 32)));
    return (unsigned)(x >> 32) == seq && (unsigned)(y >> 32) == seq;
}

__device__ __forceinline__ void flow_fail(const FlowArgs &a) {
    *reinterpret_cast<volatile int *>(a.stop) = 1;
    *a.err = 1;
}
// A warp's patience with one wait: false once it has run out, for all lanes (a
// vote at the look: what follows a wait has shuffles and votes in it).  Between
// looks at the clock and the grid's flag a poll costs one add.
struct FlowWait {
    unsigned it = 0;
    unsigned long long t0 = 0;
    __device__ __forceinline__ bool more(const FlowArgs &a) {
        if (++it < a.look) return true;
        bool out = true;
        if (a.polls == 0) {
            unsigned long long now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
            if (t0 == 0) t0 = now;
            it = 0;
            out = now - t0 > a.limit || *reinterpret_cast<volatile int *>(a.stop) != 0;
        }
        if (!__any_sync(0xffffffffu, out)) return true;
        flow_fail(a);
        return false;
    }
};

// x / d with d's reciprocal (both in the normal range): one correction step, as
// accurate as the division and a quarter of its latency.
__device__ __forceinline__ double flow_quot(double x, double d, double rd) {
    const double q = x * rd, c = fma(fma(-q, d, x), rd, q);
    // an infinite x or quotient stays one (a NaN c: exponent and a fraction bit)
    return ((unsigned)__double2hiint(c) & 0x7fffffffu) > 0x7ff00000u ? q : c;
}

__device__ __forceinline__ bool flow_ready(double x) {
    return __double2hiint(x) != -1;  // kNotReady's high word; no value that is stored has it
}

// s + the sum of M local entries a lane; false when a wait ran out (warp-uniform,
// as all below).  The first entry is polled alone: a warp
// that waits reads one word a poll and leaves the shared memory to the others.
template <int M>
__device__ __forceinline__ bool flow_local(const FlowArgs &a, const volatile double *zs,
                                           const int (&c)[kFlowFirst], const double (&v)[kFlowFirst],
                                           double &s) {
    FlowWait w;
    double x[M];
    while (x[0] = zs[c[0]], !__all_sync(0xffffffffu, flow_ready(x[0])))
        if (!w.more(a)) return false;
    if constexpr (M > 1) {
        for (;;) {
            bool all = true;
#pragma unroll
            for (int q = 1; q < M; q++) {
                x[q] = zs[c[q]];
                all = all && flow_ready(x[q]);
            }
            if (__all_sync(0xffffffffu, all)) break;
            if (!w.more(a)) return false;
        }
    }
#pragma unroll
    for (int q = 0; q < M; q++) s = fma(v[q], x[q], s);
    return true;
}

// The same for the first N values in device memory (c < 0: none).
template <int N, int C>
__device__ __forceinline__ bool flow_remote(const FlowArgs &a, const ulonglong2 *tag, const int (&c)[C],
                                            const double (&v)[C], double &s) {
    FlowWait w;
    double x[N];
    bool miss[N];
#pragma unroll
    for (int q = 0; q < N; q++) {
        x[q] = 0.0;
        miss[q] = c[q] >= 0;
    }
    for (;;) {
        bool any = false;
#pragma unroll
        for (int q = 0; q < N; q++)
            if (miss[q]) miss[q] = !flow_get(tag + c[q], a.seq, x[q]);
#pragma unroll
        for (int q = 0; q < N; q++) any = any || miss[q];
        if (!__any_sync(0xffffffffu, any)) break;
        if (!w.more(a)) return false;
    }
#pragma unroll
    for (int q = 0; q < N; q++)
        if (c[q] >= 0) s = fma(v[q], x[q], s);
    return true;
}

template <bool FWD>
__device__ __forceinline__ bool flow_item(const FlowArgs &a, const FlowTri &t, int4 it, long long ebase,
                                          int r0, int nr, double *zs, bool held, int lane) {
    const int team = it.y >> 9 & 7, cnt = (it.y & 0xff) << team, gw = it.z & 0xffff, lw = it.z >> 16;
    ulonglong2 *tag = FWD ? a.ty : a.tz;
    int row = -1;
    double s = 0.0, b = 0.0, d = 1.0, rd = 1.0;
    if (lane < cnt && (lane & ((1 << team) - 1)) == 0) {  // the row's first lane ends it
        const int at = it.x + (lane >> team);
        row = __ldg(t.rows + at);
        if (FWD) {
            b = __ldg(a.r + row);
        } else {
            flow_get(a.ty + row, a.seq, b);  // this CTA's, complete since its barrier
            d = __ldg(t.diag + at);
            rd = __ldg(t.rdiag + at);
        }
    }
    if (it.y & 256) {  // the lanes take the row's entries in turn
        const int i = __shfl_sync(0xffffffffu, row, 0), dp = __ldg(a.dpos + i);
        const int k1 = FWD ? dp : __ldg(a.rp + i + 1);
        for (int k = FWD ? __ldg(a.rp + i) : dp + 1; k < k1; k += 32 * kFlowGroup) {
            int c[kFlowGroup];
            double v[kFlowGroup];
#pragma unroll
            for (int q = 0; q < kFlowGroup; q++) {
                const int at = k + q * 32 + lane;
                c[q] = at < k1 ? __ldg(a.ci + at) : -1;
                v[q] = at < k1 ? __ldg(a.lu + at) : 0.0;
            }
            if (!flow_remote<kFlowGroup>(a, tag, c, v, s)) return false;
        }
    } else {
        // the entries of both kinds, on their way before the first wait
        const long long e = ebase + it.w + lane;
        int c[kFlowFirst], cl[kFlowFirst];
        double v[kFlowFirst], vl[kFlowFirst];
#pragma unroll
        for (int q = 0; q < kFlowFirst; q++) {
            const bool in = q < gw && lane < cnt;
            c[q] = in ? __ldg(t.ecol + e + q * cnt) : -1;
            v[q] = in ? __ldg(t.eval + e + q * cnt) : 0.0;
        }
#pragma unroll
        for (int q = 0; q < kFlowFirst; q++) {
            const bool in = q < lw && lane < cnt;
            cl[q] = in ? __ldg(t.ecol + e + (gw + q) * cnt) : -1;
            vl[q] = in ? __ldg(t.eval + e + (gw + q) * cnt) : 0.0;
            if (cl[q] < 0) cl[q] = nr;  // zs[nr] is 0, and ready
        }
        // the code for just as many: a poll's instructions are part of the hop
        if (gw > 0 && !(gw == 1   ? flow_remote<1>(a, tag, c, v, s)
                        : gw == 2 ? flow_remote<2>(a, tag, c, v, s)
                                  : flow_remote<kFlowFirst>(a, tag, c, v, s)))
            return false;
        if (lw > 0 && !(lw == 1   ? flow_local<1>(a, zs, cl, vl, s)
                        : lw == 2 ? flow_local<2>(a, zs, cl, vl, s)
                                  : flow_local<kFlowFirst>(a, zs, cl, vl, s)))
            return false;
    }
    for (int o = 1 << team >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (row >= 0) {
        s = b - s;  // one rounding at the size of b, however many entries
        if (!FWD) s = flow_quot(s, d, rd);
        if (!flow_ready(s)) s = nan("");
        if (held) *reinterpret_cast<volatile double *>(zs + (row - r0)) = s;
        flow_put(tag + row, s, a.seq);
        if (!FWD) a.z[row] = s;
    }
    return true;
}

template <bool FWD>
__device__ void flow_pass(const FlowArgs &a, const FlowTri &t, double *zs, bool held, int nr, int *ticket) {
    const int lane = threadIdx.x & 31, r0 = a.bstart[blockIdx.x];
    const int i0 = t.iptr[blockIdx.x], ni = t.iptr[blockIdx.x + 1] - i0;
    const long long ebase = t.ebase[blockIdx.x];
    auto take = [&]() {
        int q = 0;
        if (lane == 0) q = atomicAdd(ticket, 1);
        return __shfl_sync(0xffffffffu, q, 0);
    };
    // the next item is known while this one waits for its values
    int q = take();
    int4 it = q < ni ? __ldg(t.items + i0 + q) : make_int4(0, 0, 0, 0);
    while (q < ni) {
        const int qn = take();
        const int4 nx = qn < ni ? __ldg(t.items + i0 + qn) : make_int4(0, 0, 0, 0);
        if (!flow_item<FWD>(a, t, it, ebase, r0, nr, zs, held, lane)) return;
        q = qn;
        it = nx;
    }
}

__global__ void __launch_bounds__(32 * kFlowWarps, 1) k_ilu_flow(const __grid_constant__ FlowArgs a) {
    extern __shared__ double zs[];
    __shared__ int ticket[2];
    const int nr = a.bstart[blockIdx.x + 1] - a.bstart[blockIdx.x];
    const bool held = nr <= a.cap;
    if (threadIdx.x < 2) ticket[threadIdx.x] = 0;
    for (int p = 0; p < 2; p++) {
        if (held)
            for (int i = threadIdx.x; i < nr; i += blockDim.x)
                zs[i] = __longlong_as_double((long long)kNotReady);
        if (held && threadIdx.x == 0) zs[nr] = 0.0;  // what the missing entries of an item read
        __syncthreads();
        if (p == 0) flow_pass<true>(a, a.L, zs, held, nr, &ticket[0]);
        else flow_pass<false>(a, a.U, zs, held, nr, &ticket[1]);
        __syncthreads();
    }
}

// Rows grouped by level (counting sort), ascending row order inside each tier
// of a level: ELL rows (len <= kEllMax), CSR rows (<= kLongRow), CTA rows;
// n0[l], n1[l] = the first two tiers' counts.
int tier_of(int len) { return len <= kEllMax ? 0 : (len <= kLongRow ? 1 : 2); }
void group_levels(const std::vector<int> &lev, const std::vector<int> &len, int nlev,
                  std::vector<int> &rows, std::vector<int> &off, std::vector<int> &n0,
                  std::vector<int> &n1) {
    const int n = (int)lev.size();
    off.assign(nlev + 1, 0);
    for (int i = 0; i < n; i++) off[lev[i] + 1]++;
    for (int l = 0; l < nlev; l++) off[l + 1] += off[l];
    n0.assign(nlev, 0);
    n1.assign(nlev, 0);
    for (int i = 0; i < n; i++) {
        const int t = tier_of(len[i]);
        if (t == 0) n0[lev[i]]++;
        else if (t == 1) n1[lev[i]]++;
    }
    rows.resize(n);
    std::vector<int> p0(nlev), p1(nlev), p2(nlev);
    for (int l = 0; l < nlev; l++) {
        p0[l] = off[l];
        p1[l] = off[l] + n0[l];
        p2[l] = off[l] + n0[l] + n1[l];
    }
    for (int i = 0; i < n; i++) {
        const int t = tier_of(len[i]), l = lev[i];
        rows[t == 0 ? p0[l]++ : (t == 1 ? p1[l]++ : p2[l]++)] = i;
    }
}

// ELL layout of each level's first tier: width, base offsets, columns and the
// factor position of every entry (padding: the row's first entry's column,
// whose value is final before this level, with position -1 = value 0).
// Entries of row i are positions [beg(i), end(i)) of the CRS arrays.
template <typename Beg, typename End>
void build_ell(const std::vector<int> &rows, const std::vector<int> &off,
               const std::vector<int> &n0, const std::vector<int> &ci, Beg beg, End end,
               std::vector<int> &w, std::vector<long long> &eoff, std::vector<int> &ecol,
               std::vector<int> &esrc) {
    const int nl = (int)n0.size();
    w.assign(nl, 0);
    eoff.assign(nl + 1, 0);
    for (int l = 0; l < nl; l++) {
        for (int q = 0; q < n0[l]; q++) {
            const int i = rows[off[l] + q];
            w[l] = std::max(w[l], end(i) - beg(i));
        }
        eoff[l + 1] = eoff[l] + (long long)w[l] * n0[l];
    }
    ecol.assign((size_t)eoff[nl], 0);
    esrc.assign((size_t)eoff[nl], -1);
    for (int l = 0; l < nl; l++)
        for (int q = 0; q < n0[l]; q++) {
            const int i = rows[off[l] + q];
            const int b = beg(i), len = end(i) - b;
            for (int t = 0; t < w[l]; t++) {
                const long long e = eoff[l] + (long long)t * n0[l] + q;
                ecol[e] = t < len ? ci[b + t] : ci[b];
                esrc[e] = t < len ? b + t : -1;
            }
        }
}

// Rows in level order, ascending inside a level.
void level_order(const std::vector<int> &lev, int nlev, std::vector<int> &rows, std::vector<int> &off) {
    const int n = (int)lev.size();
    off.assign(nlev + 1, 0);
    for (int i = 0; i < n; i++) off[lev[i] + 1]++;
    for (int l = 0; l < nlev; l++) off[l + 1] += off[l];
    rows.resize(n);
    std::vector<int> at(off.begin(), off.end() - 1);
    for (int i = 0; i < n; i++) rows[at[lev[i]]++] = i;
}

// Rows of a CTA below which fewer CTAs do.  Where a block of R = 17 sqrt(n) rows
// (16384 at most) is half as long again as nine of ten entries (of up to 4096 rows)
// reach from the diagonal, such blocks keep more hops inside a CTA, until its 16
// warps become the bound: grids of 30^3 / 48^3 / 64^3 / 96^3 take 112 / 219 / 321 / 664
// us with 2048 rows or n / 152, 108 / 190 / 313 / 664 with 4096, 116 / 194 / 264 / 672
// with 8192, 145 / - / 280 / 611 with 16384, - / - / 454 / 855 with 24576; 1000^2 1490 /
// - / 1470 / 1396 / 1651.  A block that holds hardly one plane gains nothing (140 x
// 100 x 60: 583 us with n / 152, 621 with 15,600).  Where entries reach far, a block's
// rows wait for other blocks anyway, and more warps help: power-law rows n = 20,000
// 156 us with 2048, 118 with 1024, 88 with 256, n = 200,000 178 / 147 / 147.  Large
// blocks are for long chains (a level gives a CTA 64 rows at most), small ones for
// wide levels (64 rows and more): else 2048.
int flow_min_rows(int n, int levels, const int *rp, const int *ci) {
    const int R = (int)std::min(16384.0, 17.0 * std::sqrt((double)n)), step = std::max(1, n / 4096);
    long long near = 0, reach = 0, all = 0;
    for (int i = 0; i < n; i += step)
        for (int k = rp[i]; k < rp[i + 1]; k++) {
            const int d = std::abs(ci[k] - i);
            if (d == 0) continue;
            all++;
            near += 2 * d <= R;
            reach += 3 * d <= 2 * R;
        }
    if (10 * reach >= 9 * all) return 64LL * levels >= R ? std::max(256, R) : 2048;
    return 2 * near < all && 64LL * levels <= n ? 256 : 2048;
}

// The flow substitution's layout of one triangle (FlowTri): every block's rows
// in level order, cut into items.  The entries of row i are positions
// [beg(i), end(i)) of the CRS arrays; blocks of more than cap rows have no
// local entries.
struct FlowHost {
    std::vector<int4> items;
    std::vector<int> iptr, rows, ecol, esrc;
    std::vector<long long> ebase;
    long long longs = 0;  // entries of the rows that the warp takes from the factors
};
// Blocks [c0, c1) appended to h (their rows go to rows[bstart[c]..]).
template <typename Beg, typename End>
void flow_blocks(const std::vector<int> &lev, const std::vector<int> &bstart, int c0, int c1, int cap,
                 const int *ci, Beg beg, End end, int *rows, FlowHost &h) {
    std::vector<int> team[7], cnt, order;  // a level's rows by log2 of their lanes; 6: long
    for (int c = c0; c < c1; c++) {
        const int r0 = bstart[c], r1 = bstart[c + 1], nr = r1 - r0;
        const bool held = nr <= cap;
        int lo = nr > 0 ? lev[r0] : 0, hi = lo;
        for (int i = r0; i < r1; i++) {
            lo = std::min(lo, lev[i]);
            hi = std::max(hi, lev[i]);
        }
        order.resize(nr);
        if (hi - lo < 4 * nr + 64) {  // counting sort by level
            cnt.assign(hi - lo + 2, 0);
            for (int i = r0; i < r1; i++) cnt[lev[i] - lo + 1]++;
            for (int l = 0; l <= hi - lo; l++) cnt[l + 1] += cnt[l];
            for (int i = r0; i < r1; i++) order[cnt[lev[i] - lo]++] = i;
        } else {
            for (int i = 0; i < nr; i++) order[i] = r0 + i;
            std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return lev[x] < lev[y]; });
        }
        const size_t ebase = h.ecol.size();
        // rows of an item with a lane each: where the values of a block leave the L1
        // less than the lines that 16 warps have on their way, or every value comes
        // from device memory, smaller items wait less (96^3 grid, 5,800 rows a block,
        // items of 32 / 16 / 8: 661 / 663 / 696 us; 150^3, 22,000 rows 1377 / 1404 /
        // 1552; 160^3, 27,000 rows 2483 / 1868 / 1828; 100 x 200 x 200 1749 / 1588 /
        // 1943; 180^3, not held 3986 / 2743 / 2516)
        const int rows1 = !held ? 8 : nr > 24000 ? 16 : 32;
        for (int a = 0; a < nr;) {  // one level
            int b = a;
            for (std::vector<int> &v : team) v.clear();
            for (; b < nr && lev[order[b]] == lev[order[a]]; b++) {
                const int len = end(order[b]) - beg(order[b]);
                int g = 0;
                while (g < 6 && len > kFlowFirst << g) g++;
                team[g].push_back(order[b]);
            }
            // long rows first: they take longest
            for (int i : team[6]) {
                h.longs += end(i) - beg(i);
                rows[r0 + a] = i;
                h.items.push_back(make_int4(r0 + a++, 1 | 256 | 5 << 9, 0, 0));
            }
            for (int g = 5; g >= 0; g--) {
                const std::vector<int> &set = team[g];
                const int T = 1 << g, most = g > 0 ? 32 >> g : rows1;
                for (size_t q0 = 0; q0 < set.size(); q0 += most) {
                    const int m = (int)std::min<size_t>(most, set.size() - q0), wide = m << g;
                    int gw = 0, lw = 0;
                    for (int q = 0; q < m; q++) {
                        const int i = set[q0 + q], kb = end(i);
                        rows[r0 + a + q] = i;
                        int l = 0;
                        for (int k = beg(i); k < kb; k++) l += held && ci[k] >= r0 && ci[k] < r1;
                        gw = std::max(gw, (kb - beg(i) - l + T - 1) >> g);
                        lw = std::max(lw, (l + T - 1) >> g);
                    }
                    const size_t e = h.ecol.size();
                    h.ecol.resize(e + (size_t)(gw + lw) * wide, -1);
                    h.esrc.resize(e + (size_t)(gw + lw) * wide, -1);
                    int *ec = h.ecol.data() + e, *es = h.esrc.data() + e;
                    for (int q = 0; q < m; q++) {
                        const int i = set[q0 + q], kb = end(i);
                        int gn = 0, ln = gw << g;  // row q's entry x: lane x mod T of its T, turn x / T
                        for (int k = beg(i); k < kb; k++) {
                            const bool in = held && ci[k] >= r0 && ci[k] < r1;
                            const int x = in ? ln++ : gn++, at = (x >> g) * wide + (q << g) + (x & (T - 1));
                            ec[at] = in ? ci[k] - r0 : ci[k];
                            es[at] = k;
                        }
                    }
                    h.items.push_back(make_int4(r0 + a, m | g << 9, gw | lw << 16, (int)(e - ebase)));
                    a += m;
                }
            }
        }
        h.iptr.push_back((int)h.items.size());
        h.ebase.push_back((long long)h.ecol.size());
    }
}
// Every block, by several host threads when there are many rows; false when
// memory ran out.
template <typename Beg, typename End>
bool flow_layout(const std::vector<int> &lev, const std::vector<int> &bstart, int cap, const int *ci,
                 Beg beg, End end, FlowHost &h) {
    const int n = (int)lev.size(), G = (int)bstart.size() - 1;
    const int T = n < 100000 ? 1 : std::min({G, 8, std::max(1, (int)std::thread::hardware_concurrency())});
    std::vector<FlowHost> part(T);
    std::vector<char> ok(T, 0);
    h.rows.resize(n);
    auto work = [&](int t) {
        try {
            const int c0 = (int)((long long)G * t / T), c1 = (int)((long long)G * (t + 1) / T);
            const size_t guess = (size_t)(bstart[c1] - bstart[c0]) * 4;
            part[t].ecol.reserve(guess);
            part[t].esrc.reserve(guess);
            flow_blocks(lev, bstart, c0, c1, cap, ci, beg, end, h.rows.data(), part[t]);
            ok[t] = 1;
        } catch (...) {
        }
    };
    std::vector<std::thread> pool;
    for (int t = 1; t < T; t++) {
        try {
            pool.emplace_back(work, t);
        } catch (...) {
            work(t);
        }
    }
    work(0);
    for (auto &p : pool) p.join();
    size_t ni = 0, ne = 0;
    for (int t = 0; t < T; t++) {
        if (!ok[t]) return false;
        ni += part[t].items.size();
        ne += part[t].ecol.size();
        h.longs += part[t].longs;
    }
    h.items.reserve(ni);
    h.ecol.reserve(ne);
    h.esrc.reserve(ne);
    h.iptr.assign(1, 0);
    h.ebase.assign(1, 0);
    for (const FlowHost &p : part) {
        const int i0 = (int)h.items.size();
        const long long e0 = (long long)h.ecol.size();
        for (int v : p.iptr) h.iptr.push_back(i0 + v);
        for (long long v : p.ebase) h.ebase.push_back(e0 + v);
        h.items.insert(h.items.end(), p.items.begin(), p.items.end());
        h.ecol.insert(h.ecol.end(), p.ecol.begin(), p.ecol.end());
        h.esrc.insert(h.esrc.end(), p.esrc.begin(), p.esrc.end());
    }
    return true;
}

// Launch one substitution's levels on stream s (also used inside the capture).
template <bool FWD>
void launch_levels(const xb_plan *p, const int *d_rows, const std::vector<int> &off,
                   const std::vector<int> &n0, const std::vector<int> &n1,
                   const std::vector<int> &w, const std::vector<long long> &eoff,
                   const int *ecol, const double *eval, const double *diag, const double *r,
                   double *z, cudaStream_t s) {
    const xb::IluData &u = p->ilu;
    const int nl = (int)off.size() - 1;
    for (int l = 0; l < nl; l++) {
        const int c0 = n0[l], c1 = n1[l], c2 = off[l + 1] - off[l] - c0 - c1;
        if (c0 > 0)
            k_ilu_ell<FWD><<<(c0 + 255) / 256, 256, 0, s>>>(c0, w[l], d_rows + off[l],
                                                           ecol + eoff[l], eval + eoff[l],
                                                           diag + off[l], r, z);
        if (c1 > 0)
            k_ilu_level<FWD><<<(c1 + 255) / 256, 256, 0, s>>>(c1, d_rows + off[l] + c0, p->rowptr,
                                                             p->col, u.d_dpos, u.d_lu, r, z);
        if (c2 > 0)
            k_ilu_level_long<FWD><<<c2, 256, 0, s>>>(d_rows + off[l] + c0 + c1, p->rowptr, p->col,
                                                     u.d_dpos, u.d_lu, r, z);
    }
}

}  // namespace

namespace xb {

void ilu_free(xb_plan *p) {
    IluData &u = p->ilu;
    for (void *d : {(void *)u.d_lu, (void *)u.d_dpos, (void *)u.d_flag, (void *)u.d_in, (void *)u.d_out,
                    (void *)u.d_bstart, (void *)u.d_ty, (void *)u.d_tz, (void *)u.d_stop,
                    (void *)u.d_lrows, (void *)u.d_urows, (void *)u.d_lecol, (void *)u.d_uecol,
                    (void *)u.d_leval, (void *)u.d_ueval, (void *)u.d_udiag})
        cudaFree(d);
    for (IluData::Flow *f : {&u.fl, &u.fu})
        for (void *d : {(void *)f->d_items, (void *)f->d_iptr, (void *)f->d_ebase, (void *)f->d_rows,
                        (void *)f->d_ecol, (void *)f->d_eval, (void *)f->d_diag, (void *)f->d_rdiag})
            cudaFree(d);
    if (u.exec) cudaGraphExecDestroy(u.exec);
    if (u.graph) cudaGraphDestroy(u.graph);
    u = IluData();
}

int ilu_levels(int n, const int *rp, const int *ci, std::vector<int> &dpos, std::vector<int> &lev,
               std::vector<int> &ulev, int *nl, int *nu) {
    dpos.assign(n, 0);
    lev.assign(n, 0);
    ulev.assign(n, 0);
    *nl = n > 0 ? 1 : 0;
    *nu = n > 0 ? 1 : 0;
    for (int i = 0; i < n; i++) {
        int d = -1, m = -1;
        for (int q = rp[i]; q < rp[i + 1]; q++) {
            const int k = ci[q];
            if (k < i) m = std::max(m, lev[k]);
            else if (k == i) d = q;
        }
        if (d < 0) return set_error(XB_EBREAKDOWN, "ILU(0): row %d has no diagonal entry", i);
        dpos[i] = d;
        lev[i] = m + 1;
        *nl = std::max(*nl, lev[i] + 1);
    }
    for (int i = n - 1; i >= 0; i--) {
        int m = -1;
        for (int q = dpos[i] + 1; q < rp[i + 1]; q++) m = std::max(m, ulev[ci[q]]);
        ulev[i] = m + 1;
        *nu = std::max(*nu, ulev[i] + 1);
    }
    return XB_OK;
}

namespace {

// Device memory that the preconditioner keeps.
template <typename T>
int keep(IluData &u, T **d, size_t bytes) {
    XB_CUDA(cudaMalloc(d, std::max<size_t>(8, bytes)));
    u.bytes += (double)bytes;
    return XB_OK;
}

int upload(int **d, const std::vector<int> &h, cudaStream_t s, IluData *u = nullptr) {
    if (u) XB_TRY(keep(*u, d, h.size() * 4));
    else XB_CUDA(cudaMalloc(d, std::max<size_t>(1, h.size()) * 4));
    if (!h.empty()) XB_CUDA(cudaMemcpyAsync(*d, h.data(), h.size() * 4, cudaMemcpyHostToDevice, s));
    return XB_OK;
}

// ELL values of a layout's entries from the factors.
int fill_entries(IluData &u, double **val, const std::vector<int> &src, cudaStream_t s) {
    int *d_src = nullptr;
    XB_TRY(keep(u, val, src.size() * sizeof(double)));
    XB_TRY(upload(&d_src, src, s));
    if (!src.empty()) {
        k_ell_fill<<<(unsigned)((src.size() + 255) / 256), 256, 0, s>>>((long long)src.size(), d_src, u.d_lu, *val);
        XB_LAUNCHED("k_ell_fill");
    }
    cudaFree(d_src);  // waits for the kernel
    return XB_OK;
}

int upload_flow(IluData &u, IluData::Flow &f, const FlowHost &h, cudaStream_t s) {
    static_assert(sizeof(int4) == 16 && sizeof(long long) == 8, "layout");
    XB_TRY(keep(u, &f.d_items, h.items.size() * sizeof(int4)));
    XB_CUDA(cudaMemcpyAsync(f.d_items, h.items.data(), h.items.size() * sizeof(int4), cudaMemcpyHostToDevice, s));
    XB_TRY(keep(u, &f.d_ebase, h.ebase.size() * sizeof(long long)));
    XB_CUDA(cudaMemcpyAsync(f.d_ebase, h.ebase.data(), h.ebase.size() * sizeof(long long),
                            cudaMemcpyHostToDevice, s));
    XB_TRY(upload(&f.d_iptr, h.iptr, s, &u));
    XB_TRY(upload(&f.d_rows, h.rows, s, &u));
    XB_TRY(upload(&f.d_ecol, h.ecol, s, &u));
    u.flow_bytes += 16.0 * h.items.size() + 4.0 * h.rows.size() + 12.0 * h.ecol.size();
    return fill_entries(u, &f.d_eval, h.esrc, s);
}

int rows_host(xb_plan *p, std::vector<int> &ci) {
    ci.resize(p->nnz);
    if (p->nnz > 0) XB_CUDA(cudaMemcpy(ci.data(), p->col, (size_t)p->nnz * 4, cudaMemcpyDeviceToHost));
    return XB_OK;
}

// The level launches of both substitutions (path 0), captured once: built when
// that path is first taken.
int ensure_graph(xb_plan *p, cudaStream_t s) {
    IluData &u = p->ilu;
    if (u.exec) return XB_OK;
    const int n = p->n;
    const std::vector<int> &rp = p->h_rowptr;
    std::vector<int> ci, dpos, lev, ulev;
    int nl = 0, nu = 0;
    XB_TRY(rows_host(p, ci));
    XB_TRY(ilu_levels(n, rp.data(), ci.data(), dpos, lev, ulev, &nl, &nu));
    std::vector<int> llen(n), ulen(n);
    for (int i = 0; i < n; i++) {
        llen[i] = dpos[i] - rp[i];
        ulen[i] = rp[i + 1] - dpos[i] - 1;
    }
    std::vector<int> lrows, urows, loff, uoff, ln0, ln1, un0, un1, lw, uw, lecol, lesrc, uecol, uesrc;
    std::vector<long long> leoff, ueoff;
    group_levels(lev, llen, nl, lrows, loff, ln0, ln1);
    group_levels(ulev, ulen, nu, urows, uoff, un0, un1);
    build_ell(lrows, loff, ln0, ci, [&](int i) { return rp[i]; }, [&](int i) { return dpos[i]; }, lw,
              leoff, lecol, lesrc);
    build_ell(urows, uoff, un0, ci, [&](int i) { return dpos[i] + 1; },
              [&](int i) { return rp[i + 1]; }, uw, ueoff, uecol, uesrc);
    for (int **d : {&u.d_lrows, &u.d_urows, &u.d_lecol, &u.d_uecol}) {
        cudaFree(*d);
        *d = nullptr;
    }
    for (double **d : {&u.d_leval, &u.d_ueval, &u.d_udiag, &u.d_out}) {
        cudaFree(*d);
        *d = nullptr;
    }
    XB_TRY(upload(&u.d_lrows, lrows, s, &u));
    XB_TRY(upload(&u.d_urows, urows, s, &u));
    XB_TRY(upload(&u.d_lecol, lecol, s, &u));
    XB_TRY(upload(&u.d_uecol, uecol, s, &u));
    XB_TRY(fill_entries(u, &u.d_leval, lesrc, s));
    XB_TRY(fill_entries(u, &u.d_ueval, uesrc, s));
    XB_TRY(keep(u, &u.d_udiag, (size_t)n * sizeof(double)));
    XB_TRY(keep(u, &u.d_out, (size_t)n * sizeof(double)));
    k_diag_fill<<<(n + 255) / 256, 256, 0, s>>>(n, u.d_urows, u.d_dpos, u.d_lu, u.d_udiag, nullptr,
                                                nullptr);
    XB_LAUNCHED("k_diag_fill");
    cudaStream_t cs = nullptr;
    XB_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        launch_levels<true>(p, u.d_lrows, loff, ln0, ln1, lw, leoff, u.d_lecol, u.d_leval, u.d_udiag,
                            u.d_in, u.d_out, cs);
        launch_levels<false>(p, u.d_urows, uoff, un0, un1, uw, ueoff, u.d_uecol, u.d_ueval, u.d_udiag,
                             u.d_out, u.d_out, cs);
        e = cudaStreamEndCapture(cs, &u.graph);
    }
    cudaStreamDestroy(cs);
    if (e == cudaSuccess) e = cudaGraphInstantiate(&u.exec, u.graph, 0);
    if (e != cudaSuccess) return cuda_error(e, "ILU(0): capture of the substitutions");
    XB_CUDA(cudaStreamSynchronize(s));
    return XB_OK;
}

}  // namespace

int ensure_ilu(xb_plan *p, cudaStream_t s) {
    if (!p->subs.empty())
        return set_error(XB_EINVAL, "ILU(0): not available for a plan split into row blocks");
    IluData &u = p->ilu;
    if (u.built) return u.status == XB_OK ? XB_OK : set_error(u.status, "ILU(0): zero pivot");
    if (p->sym) return set_error(XB_EINVAL, "ILU(0) needs full (general) CRS storage");
    ilu_free(p);  // a build that failed half-way left nothing usable
    const int n = p->n, nnz = p->nnz;
    const std::vector<int> &rp = p->h_rowptr;
    std::vector<int> ci, dpos, lev, ulev, lorder, loff;
    int nl = 0, nu = 0;
    XB_TRY(rows_host(p, ci));
    XB_TRY(ilu_levels(n, rp.data(), ci.data(), dpos, lev, ulev, &nl, &nu));
    level_order(lev, nl, lorder, loff);
    // factors, level by level
    int *d_order = nullptr;
    XB_TRY(upload(&u.d_dpos, dpos, s, &u));
    XB_TRY(upload(&d_order, lorder, s));
    XB_TRY(keep(u, &u.d_lu, (size_t)nnz * sizeof(double)));
    XB_TRY(keep(u, &u.d_flag, 2 * sizeof(int)));  // zero pivot; pivot out of the flow path's range
    XB_TRY(keep(u, &u.d_in, (size_t)n * sizeof(double)));
    XB_CUDA(cudaMemsetAsync(u.d_flag, 0, 2 * sizeof(int), s));
    if (nnz > 0)
        XB_CUDA(cudaMemcpyAsync(u.d_lu, p->val, (size_t)nnz * sizeof(double),
                                cudaMemcpyDeviceToDevice, s));
    for (int l = 0; l < nl; l++) {
        const int cnt = loff[l + 1] - loff[l];
        if (cnt == 0) continue;
        const int wpb = 8;  // warps per CTA
        k_ilu_factor<<<(cnt + wpb - 1) / wpb, 32 * wpb, 0, s>>>(
            cnt, d_order + loff[l], p->rowptr, p->col, u.d_dpos, u.d_lu, u.d_flag);
    }
    XB_LAUNCHED("k_ilu_factor");
    int dev = 0, coop = 0, smem = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (coop && n > 0) {  // the flow layout, while the factorization runs
        const int cap = (smem - 1024) / 8 - 1;
        const int least = flow_min_rows(n, std::max(nl, nu), rp.data(), ci.data());
        const int G = std::max(1, std::min(num_sms(), (n + least - 1) / least));
        std::vector<int> bstart(G + 1, n);
        bstart[0] = 0;
        const double total = (double)nnz + 4.0 * n;  // blocks of about equal work
        for (int i = 0, c = 0; i < n && c + 1 < G; i++)
            while (c + 1 < G && (double)rp[i] + 4.0 * i >= total * (c + 1) / G) bstart[++c] = i;
        for (int c = 1; c <= G; c++) u.maxrows = std::max(u.maxrows, bstart[c] - bstart[c - 1]);
        u.cap = std::min(u.maxrows, cap);
        FlowHost hl, hu;
        if (!flow_layout(lev, bstart, cap, ci.data(), [&](int i) { return rp[i]; },
                         [&](int i) { return dpos[i]; }, hl) ||
            !flow_layout(ulev, bstart, cap, ci.data(), [&](int i) { return dpos[i] + 1; },
                         [&](int i) { return rp[i + 1]; }, hu)) {
            cudaStreamSynchronize(s);
            cudaFree(d_order);
            return set_error(XB_ENOMEM, "ILU(0): host memory for the substitutions' layout");
        }
        XB_TRY(upload(&u.d_bstart, bstart, s, &u));
        XB_TRY(upload_flow(u, u.fl, hl, s));
        XB_TRY(upload_flow(u, u.fu, hu, s));
        // r in, z out, the pivots and reciprocals, both triangles' published values
        // out and the first one's in again
        u.flow_bytes += 12.0 * (hl.longs + hu.longs) + (8.0 + 8.0 + 16.0 + 32.0 + 16.0) * n;
        XB_TRY(keep(u, &u.fu.d_diag, (size_t)n * sizeof(double)));
        XB_TRY(keep(u, &u.fu.d_rdiag, (size_t)n * sizeof(double)));
        k_diag_fill<<<(n + 255) / 256, 256, 0, s>>>(n, u.fu.d_rows, u.d_dpos, u.d_lu, u.fu.d_diag,
                                                    u.fu.d_rdiag, u.d_flag + 1);
        XB_LAUNCHED("k_diag_fill");
        XB_TRY(keep(u, &u.d_ty, (size_t)n * 16));
        XB_TRY(keep(u, &u.d_tz, (size_t)n * 16));
        XB_TRY(keep(u, &u.d_stop, sizeof(int)));
        XB_CUDA(cudaMemsetAsync(u.d_ty, 0, (size_t)n * 16, s));
        XB_CUDA(cudaMemsetAsync(u.d_tz, 0, (size_t)n * 16, s));
        XB_CUDA(cudaMemsetAsync(u.d_stop, 0, sizeof(int), s));
        XB_CUDA(cudaFuncSetAttribute(k_ilu_flow, cudaFuncAttributeMaxDynamicSharedMemorySize, smem - 1024));
        u.grid = G;
        u.limit_ns = 2000000000ull + 2000ull * (nl + nu);
    }
    int flag[2] = {0, 0};
    XB_CUDA(cudaMemcpyAsync(flag, u.d_flag, sizeof flag, cudaMemcpyDeviceToHost, s));
    XB_CUDA(cudaStreamSynchronize(s));
    cudaFree(d_order);
    u.built = true;
    u.status = flag[0] ? XB_EBREAKDOWN : XB_OK;
    if (flag[1]) u.grid = 0;  // the graph path divides
    if (flag[0]) return set_error(XB_EBREAKDOWN, "ILU(0): zero pivot");
    return XB_OK;
}

// Which substitution to run: the flow launch, faster on every pattern measured
// (k_ilu_flow), or (0) the captured graph of level launches, where there is no
// cooperative launch or a pivot's reciprocal leaves the normal range.
// XB_ILU_MODE=0/1 forces one.
int ilu_mode(const xb_plan *p) {
    static const int env = [] {
        const char *e = std::getenv("XB_ILU_MODE");
        return e ? std::atoi(e) : -1;
    }();
    if (p->ilu.grid == 0) return 0;
    if (p->ilu_mode >= 0) return p->ilu_mode;
    return env >= 0 ? env : 1;
}

int ilu_check(xb_plan *p, cudaStream_t s) {
    volatile int *err = reinterpret_cast<volatile int *>(p->h_pin + 61);
    if (!*err) return XB_OK;
    *err = 0;
    if (p->ilu.d_stop) {
        XB_CUDA(cudaMemsetAsync(p->ilu.d_stop, 0, sizeof(int), s));
        XB_CUDA(cudaStreamSynchronize(s));  // the next application may be on another stream
    }
    return set_error(XB_ETIMEOUT, "ILU(0): a wait for another row's value ran out");
}

int ilu_apply(xb_plan *p, const double *r, double *z, cudaStream_t s) {
    IluData &u = p->ilu;
    XB_TRY(ensure_ilu(p, s));
    if (p->n == 0) return XB_OK;
    const size_t bytes = (size_t)p->n * sizeof(double);
    if (ilu_mode(p) == 1) {
        const uintptr_t ra = (uintptr_t)r, za = (uintptr_t)z;
        if (ra < za + bytes && za < ra + bytes) {  // overlapping operands: rows of r are read late
            XB_CUDA(cudaMemcpyAsync(u.d_in, r, bytes, cudaMemcpyDeviceToDevice, s));
            r = u.d_in;
        }
        auto tri = [](const IluData::Flow &f) {
            return FlowTri{reinterpret_cast<const int4 *>(f.d_items), f.d_iptr, f.d_ebase, f.d_rows,
                           f.d_ecol, f.d_eval, f.d_diag, f.d_rdiag};
        };
        FlowArgs a{};
        a.L = tri(u.fl);
        a.U = tri(u.fu);
        a.bstart = u.d_bstart;
        a.rp = p->rowptr;
        a.ci = p->col;
        a.dpos = u.d_dpos;
        a.lu = u.d_lu;
        a.r = r;
        a.z = z;
        a.ty = reinterpret_cast<ulonglong2 *>(u.d_ty);
        a.tz = reinterpret_cast<ulonglong2 *>(u.d_tz);
        if (++u.seq == 0) u.seq = 1;
        a.seq = u.seq;
        a.polls = (unsigned)p->ilu_polls;
        a.look = a.polls ? a.polls : 64u;
        a.limit = u.limit_ns;
        a.err = reinterpret_cast<volatile int *>(p->h_pin + 61);
        a.stop = u.d_stop;
        a.cap = u.cap;
        void *args[] = {&a};
        XB_CUDA(cudaLaunchCooperativeKernel((const void *)k_ilu_flow, u.grid, 32 * kFlowWarps, args,
                                            (size_t)(u.cap + 1) * sizeof(double), s));
        return XB_OK;
    }
    XB_TRY(ensure_graph(p, s));
    XB_CUDA(cudaMemcpyAsync(u.d_in, r, bytes, cudaMemcpyDeviceToDevice, s));
    XB_CUDA(cudaGraphLaunch(u.exec, s));
    XB_CUDA(cudaMemcpyAsync(z, u.d_out, bytes, cudaMemcpyDeviceToDevice, s));
    return XB_OK;
}

double ilu_apply_bytes(const xb_plan *p) {
    if (ilu_mode(p) == 1) return p->ilu.flow_bytes;
    // the graph of level launches: both triangles once (value + column), rowptr and diagonal positions
    // twice, r read, z written by the forward pass, read and written by the
    // backward pass, and each row's level slot twice
    const double n = p->n, nnz = p->nnz;
    return 12.0 * nnz + 2.0 * 4.0 * (n + 1) + 2.0 * 4.0 * n + 8.0 * n * 4.0 + 2.0 * 4.0 * n +
           32.0 * n;  // + copies into and out of the captured solve's buffers
}

}  // namespace xb

extern "C" {

int xb_ilu0_setup(xb_plan *p, void *stream) {
    if (!p) return xb::set_error(XB_EINVAL, "ilu0_setup: NULL plan");
    return xb::ensure_ilu(p, (cudaStream_t)stream);
}

int xb_ilu0_apply(xb_plan *p, const double *r, double *z, void *stream) {
    if (!p || (p->n > 0 && (!r || !z)) || r == z)
        return xb::set_error(XB_EINVAL, "ilu0_apply: bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    XB_TRY(xb::ilu_apply(p, r, z, s));
    XB_CUDA(cudaStreamSynchronize(s));
    return xb::ilu_check(p, s);
}

int xb_ilu0_config(xb_plan *p, int32_t mode, int32_t barrier_polls) {
    if (!p || mode < -1 || mode > 1 || barrier_polls < 0)
        return xb::set_error(XB_EINVAL, "ilu0_config: plan %p mode %d polls %d", (void *)p, mode,
                             barrier_polls);
    p->ilu_mode = mode;
    p->ilu_polls = barrier_polls;
    return XB_OK;
}

int xb_ilu0_factors(xb_plan *p, double *lu, void *stream) {
    if (!p || (p->nnz > 0 && !lu)) return xb::set_error(XB_EINVAL, "ilu0_factors: bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    XB_TRY(xb::ensure_ilu(p, s));
    if (p->nnz > 0)
        XB_CUDA(cudaMemcpyAsync(lu, p->ilu.d_lu, (size_t)p->nnz * sizeof(double),
                                cudaMemcpyDeviceToDevice, s));
    return XB_OK;
}

}  // extern "C"

extern "C" int xb_ilu_levels(int32_t n, const int32_t *rowptr, const int32_t *col, int32_t *lev,
                             int32_t *ulev, int32_t *nlevels) {
    if (n < 0 || !rowptr || (n > 0 && !col))
        return xb::set_error(XB_EINVAL, "ilu_levels: bad argument");
    std::vector<int> d, l, u;
    int nl = 0, nu = 0;
    XB_TRY(xb::ilu_levels(n, rowptr, col, d, l, u, &nl, &nu));
    if (lev) std::copy(l.begin(), l.end(), lev);
    if (ulev) std::copy(u.begin(), u.end(), ulev);
    if (nlevels) {
        nlevels[0] = nl;
        nlevels[1] = nu;
    }
    return XB_OK;
}
