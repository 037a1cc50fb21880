// One orthogonalisation of the Arnoldi process (Sec. 3.2.2: MGS, CGS, DGKS,
// BCGS) as one cooperative launch of clusters.
//
// CTA c owns the elements [c * chunk, (c + 1) * chunk) of w and of every basis
// row.  Its part of w stays in shared memory from the first dot product to the
// last update when it fits.  A producer warp streams the basis rows through a
// ring of shared-memory stages with bulk copies, so the rows that follow an
// exchange are on the chip before the exchange ends.  The inner products are
// summed over the grid with one exchange per block of rows instead of one
// launch per row.
#include "krylov.cuh"
#include "perdevice.cuh"

#include <algorithm>

namespace {

constexpr int kGsMaxClusters = 96;   // clusters one exchange has room for
constexpr int kGsVals = 64;          // values of one exchange
constexpr int kGsMaxK = 512;         // basis rows
constexpr int kGsMaxStages = 8;
constexpr int kGsSlotsAt = 128;      // words of d_ticket before the grid's exchange slots
constexpr size_t kGsSlotBytes = sizeof(ulonglong2) * 2 * kGsVals * kGsMaxClusters;
constexpr long long kGsWait = 4000000000LL;  // cycles (~2 s) after which a wait gives up

template <typename VB>
struct GsArgs {
    int64_t n, ld, chunk;
    const VB *V;
    VB *w;
    xb::GmDev st;         // misc null: a plain sweep (unit scales, never stopped)
    double *col;          // column j: h_0..h_j, then ||w||
    int j, method, cs, stages;
    unsigned base;        // this launch's exchanges have the numbers base + 1, base + 2, ..
    unsigned *stop;       // a wait of the grid ran out
    unsigned polls, look; // polls of one wait (0: the clock decides); polls between looks
    ulonglong2 *slots;    // 2 x kGsVals x kGsMaxClusters
    int *err;             // host-visible: a wait ran out
    unsigned long long *late, tag;  // host-visible words: 4 tag + GM_STOP after step tag
};

// ---- values that carry their exchange number ------------------------------------
// A double travels as two 8-byte words, each with the number of its exchange:
// a reader that sees the number in both has the whole value, whatever order
// the words arrive in, and no fence or flag is needed.  A slot that was never
// written has number 0, which no exchange has (gs_numbers).
__device__ __forceinline__ void pack(double v, unsigned seq, unsigned long long &x,
                                     unsigned long long &y) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned long long s = (unsigned long long)seq << 32;
    x = s | (b & 0xffffffffu);
    y = s | (b >> 32);
}
__device__ __forceinline__ bool unpack(unsigned long long x, unsigned long long y, unsigned seq,
                                       double &v) {
    v = __longlong_as_double((long long)((x & 0xffffffffu) | (y << 32)));
    return (unsigned)(x >> 32) == seq && (unsigned)(y >> 32) == seq;
}
__device__ __forceinline__ void put_global(ulonglong2 *p, double v, unsigned seq) {
    unsigned long long x, y;
    pack(v, seq, x, y);
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(x), "l"(y) : "memory");
}
__device__ __forceinline__ bool get_global(const ulonglong2 *p, unsigned seq, double &v) {
    unsigned long long x, y;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
    return unpack(x, y, seq, v);
}
__device__ __forceinline__ void put_cluster(unsigned addr, int rank, double v, unsigned seq) {
    unsigned long long x, y;
    unsigned r;
    pack(v, seq, x, y);
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    asm volatile("st.relaxed.cluster.shared::cluster.v2.b64 [%0], {%1, %2};" ::"r"(r), "l"(x), "l"(y)
                 : "memory");
}
__device__ __forceinline__ bool get_shared(unsigned addr, unsigned seq, double &v) {
    unsigned long long x, y;
    asm volatile("ld.relaxed.cluster.shared::cta.v2.b64 {%0, %1}, [%2];"
                 : "=l"(x), "=l"(y) : "r"(addr) : "memory");
    return unpack(x, y, seq, v);
}

// ---- synchronisation --------------------------------------------------------------
__device__ __forceinline__ unsigned sptr(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// The same barrier; true in every thread when some thread's flag is set.
__device__ __forceinline__ bool bar_any(int id, int threads, bool flag) {
    unsigned r;
    asm volatile("{\n.reg .pred p, q;\n"
                 "setp.ne.u32 p, %3, 0;\n"
                 "bar.red.or.pred q, %1, %2, p;\n"
                 "selp.b32 %0, 1, 0, q;\n}"
                 : "=r"(r) : "r"(id), "r"(threads), "r"((unsigned)flag) : "memory");
    return r != 0;
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
    __threadfence_block();
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n"
                 "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ int cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}
__device__ __forceinline__ int cluster_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return (int)r;
}
__device__ __forceinline__ void mbar_init(unsigned bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_done(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile("{\n.reg .pred p;\n"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                 "selp.b32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void bulk_copy(unsigned dst, const void *src, unsigned bytes, unsigned bar,
                                          uint64_t policy) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
                 "[%0], [%1], %2, [%3], %4;" ::"r"(dst), "l"(src), "r"(bytes), "r"(bar), "l"(policy)
                 : "memory");
}

// A bounded wait: expired() is true once the wait has lasted kGsWait cycles, or
// as many polls as the caller allows, or another wait of the grid has run out.
// Between looks at the clock and the grid's flag a poll costs one add (look: the
// polls between them, in a register).
struct Patience {
    unsigned it = 0;
    long long t0 = 0;
    template <typename VB>
    __device__ __forceinline__ bool expired(const GsArgs<VB> &a, unsigned look) {
        if (++it < look) return false;
        if (a.polls != 0) return true;
        it = 0;
        const long long now = clock64();
        if (t0 == 0) t0 = now;
        return now - t0 > kGsWait || *reinterpret_cast<const volatile unsigned *>(a.stop) != 0u;
    }
};

// Sums NV per-lane values over the warp: v[0] of lane l is the total of value
// l / (32 / NV).  Each step halves the values a lane carries, so it takes
// NV - 1 + log2(32 / NV) adds instead of 5 NV: an FP64 add holds the pipe of
// an SM quarter for ~80 cycles whatever it adds.
template <int NV>
__device__ __forceinline__ void warp_totals(double (&v)[NV], int lane) {
    int o = 16;
#pragma unroll
    for (int h = NV / 2; h >= 1; h /= 2) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < h; i++) {
            const double send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        o >>= 1;
    }
    for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
}

// GRAM: the rows' own products that a kernel takes, 0 none, 1 the newest row's, 2
// all pairs of a block.  BCGS, CGS and DGKS take none: in FP64 one kernel has both
// kinds of passes (apart, BCGS took 1.5% longer), in FP32 CGS and DGKS have their own
// (together, BCGS took 0.4% longer).
constexpr int kCgs = 3;
constexpr int gram_count(int kb, int gram) {
    return gram == 1 ? kb - 1 : (gram == 2 ? kb * (kb - 1) / 2 : 0);
}

// Chains of a thread's FP32 partial sums: 13 terms each at n = 2.1M, 7 for MGS (where
// their errors enter the corrections too), then FP64 takes over.
template <typename VB, int KB, int GRAM>
constexpr int chains() { return sizeof(VB) == 4 ? (KB <= 4 && GRAM == 1 ? 8 : 4) : 1; }

// Launch shape: NT = 256 compute threads, two warps on each quarter of the SM
// (one waits or loads while the other's FMAs hold the FP64 pipe; more would only
// add to the sums over threads), or 512 where the passes are long and w comes
// from device memory, whose latency eight warps do not hide.
template <typename VB, int KB, int NT>
constexpr int gs_elems() {  // per thread and tile
    return sizeof(VB) == 4 ? (KB <= 4 ? 8 : 4) : (KB == 2 && NT == 256 ? 4 : 2);
}
template <typename VB, int KB, int NT>
constexpr int gs_tile() { return NT * gs_elems<VB, KB, NT>(); }
template <typename VB, int KB, int NT>
constexpr int gs_pitch() { return gs_tile<VB, KB, NT>() * (int)sizeof(VB) + 16; }
// Shared memory besides w and the stages: exchange slots.
template <int NT>
constexpr int gs_xch_bytes() { return 2 * kGsVals * (NT / 32) * 16 + 2 * kGsVals * 16; }

template <typename VB, int KB, int NT>
struct GsShared {
    unsigned long long full[kGsMaxStages], empty[kGsMaxStages];
    double hcol[kGsMaxK + 1];
    VB cf[kGsMaxK];                               // CGS, DGKS: one for the CTA
    VB cfw[NT / 32][KB];            // block methods: one for each warp
    int abort;
};

// The CTA's state: everything the roles share.
template <typename VB, int KB, int NT>
struct Ctx {
    GsShared<VB, KB, NT> *S;
    const GsArgs<VB> *a;
    const VB *Vc;          // basis, from the CTA's first element
    unsigned ring;         // stages
    unsigned part, bc;     // exchange slots: partial sums of the cluster, totals
    unsigned row0, pitch;  // low words of Vc and of a row's bytes (alignment)
    int len, tiles, rank, lane, wv;
    unsigned look;
    int st, ph;            // ring position: stage, and times the ring went round
    int pass;              // odd passes take the tiles from the end: they start on the
                           // lines the previous one left in L2
    bool fine;
    __device__ __forceinline__ void next() {
        if (++st == a->stages) {
            st = 0;
            ph++;
        }
    }
};

template <typename VB, int KB, int NT>
__device__ __forceinline__ void give_up(Ctx<VB, KB, NT> &c) {
    *reinterpret_cast<volatile int *>(&c.S->abort) = 1;
    *reinterpret_cast<volatile unsigned *>(c.a->stop) = 1u;
    *reinterpret_cast<volatile int *>(c.a->err) = 1;
    c.fine = false;
}

// Waits for a stage.  A lane that gives up, or sees that another has, goes on with
// what is there, beside the lanes that need not (the addresses stay those of the
// stage): nothing branches on one lane's c.fine before a vote has made it the
// warp's.
template <typename VB, int KB, int NT>
__device__ __forceinline__ void wait_bar(Ctx<VB, KB, NT> &c, unsigned bar, unsigned parity) {
    Patience w;
    while (c.fine && !mbar_done(bar, parity)) {
        if (*reinterpret_cast<volatile int *>(&c.S->abort)) c.fine = false;
        else if (w.expired(*c.a, c.look)) give_up(c);
    }
}

// ---- producer ---------------------------------------------------------------------
// One unit: rows row0 .. row0 + nr - 1 of tile t.  The copies take whole 16-byte
// blocks: an end that lies inside one belongs to the same allocation.
template <typename VB, int KB, int NT>
__device__ __forceinline__ void produce(Ctx<VB, KB, NT> &c, int t, int row0, int nr, uint64_t policy) {
    if (!c.fine) return;
    const unsigned full = sptr(&c.S->full[c.st]);
    if (c.ph > 0) {
        // a consumer that gave up has said so before it freed a stage that may
        // still be filling
        wait_bar(c, sptr(&c.S->empty[c.st]), (c.ph - 1) & 1);
        c.fine = __all_sync(0xffffffffu, c.fine && !*reinterpret_cast<volatile int *>(&c.S->abort));
        if (!c.fine) return;
    }
    constexpr int T = gs_tile<VB, KB, NT>();
    const int cnt = min(T, c.len - t * T);
    uintptr_t lo = 0, hi = 0;
    if (c.lane < nr) {
        lo = (uintptr_t)(c.Vc + (int64_t)(row0 + c.lane) * c.a->ld + (int64_t)t * T);
        hi = (lo + cnt * sizeof(VB) + 15) & ~(uintptr_t)15;
        lo &= ~(uintptr_t)15;
    }
    const unsigned bytes = __reduce_add_sync(0xffffffffu, (unsigned)(hi - lo));
    if (c.lane == 0) mbar_expect(full, bytes);
    __syncwarp();
    if (c.lane < nr)
        bulk_copy(c.ring + (c.st * KB + c.lane) * gs_pitch<VB, KB, NT>(), (const void *)lo,
                  (unsigned)(hi - lo), full, policy);
    c.next();
}

// Waits for the copies that are in flight: the consumers of a sweep that is given
// up leave them behind, and a CTA must not end before its copies.
template <typename VB, int KB, int NT>
__device__ void drain(Ctx<VB, KB, NT> &c) {
    for (int i = 0; i < c.a->stages; i++) {
        const int ph = i < c.st ? c.ph : c.ph - 1;  // the stage's last use
        if (ph < 0) continue;
        for (unsigned it = 0; it < (1u << 22) && !mbar_done(sptr(&c.S->full[i]), ph & 1); it++) {
        }
    }
}

// ---- consumers --------------------------------------------------------------------
template <typename VB, int KB, int NT>
__device__ __forceinline__ void unit_wait(Ctx<VB, KB, NT> &c) {
    wait_bar(c, sptr(&c.S->full[c.st]), c.ph & 1);
}
template <typename VB, int KB, int NT>
__device__ __forceinline__ void unit_free(Ctx<VB, KB, NT> &c) {
    __syncwarp();
    if (c.lane == 0) mbar_arrive(sptr(&c.S->empty[c.st]));
    c.next();
}
// Address of row r of the current unit (rows whose start is not 16-byte aligned
// sit at their offset in the block; tiles are whole blocks).
template <typename VB, int KB, int NT>
__device__ __forceinline__ unsigned unit_row(const Ctx<VB, KB, NT> &c, int first, int r) {
    return c.ring + (c.st * KB + r) * gs_pitch<VB, KB, NT>() + ((c.row0 + (unsigned)(first + r) * c.pitch) & 15u);
}
// A thread's E values of a row of the unit: FP64 NT apart (a row may start at
// any 8-byte offset), FP32 four together in one 16-byte load (the solvers' FP32
// rows are aligned).
template <typename VB, int E, int NT>
constexpr int place(int tid, int i) {
    return sizeof(VB) == 4 ? 4 * tid + i % 4 + i / 4 * 4 * NT : tid + i * NT;
}
template <int NT, int E>
__device__ __forceinline__ void lds_row(unsigned a, double (&v)[E]) {
#pragma unroll
    for (int i = 0; i < E; i++)
        asm volatile("ld.shared::cta.f64 %0, [%1];" : "=d"(v[i]) : "r"(a + i * NT * 8));
}
template <int NT, int E>
__device__ __forceinline__ void lds_row(unsigned a, float (&v)[E]) {
    static_assert(E % 4 == 0, "16-byte loads");
#pragma unroll
    for (int i = 0; i < E; i += 4)
        asm volatile("ld.shared::cta.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[i]), "=f"(v[i + 1]), "=f"(v[i + 2]), "=f"(v[i + 3])
                     : "r"(a + i * NT * 4));
}

// One tile of a pass; FULL: every thread has all its elements.
template <typename VB, int KB, int NT, int GRAM, bool GR, bool FIN, bool FULL, int NA, int E>
__device__ __forceinline__ void gs_tile_pass(Ctx<VB, KB, NT> &c, int e0, VB (&x)[E], VB *dst, int u0, int nu,
                                             const VB *cf, int d0, int nd, VB (&acc)[NA][chains<VB, KB, GRAM>()]) {
    constexpr int AW = chains<VB, KB, GRAM>();
    const int tid = threadIdx.x;
    const unsigned off = place<VB, E, NT>(tid, 0) * (int)sizeof(VB);
    for (int i0 = 0; i0 < nu; i0 += KB) {
        unit_wait(c);
        const int nr = min(KB, nu - i0);
#pragma unroll
        for (int r = 0; r < KB; r++) {
            if (r < nr) {
                VB v[E];
                lds_row<NT>(unit_row(c, u0 + i0, r) + off, v);
                const VB cr = cf[i0 + r];
#pragma unroll
                for (int i = 0; i < E; i++) x[i] = fma(-cr, v[i], x[i]);
            }
        }
        unit_free(c);
    }
    if (dst) {
#pragma unroll
        for (int i = 0; i < E; i++)
            if (FULL || e0 + place<VB, E, NT>(tid, i) < c.len) dst[e0 + place<VB, E, NT>(tid, i)] = x[i];
    }
    if constexpr (FIN) {
#pragma unroll
        for (int i = 0; i < E; i++)
            if (FULL || e0 + place<VB, E, NT>(tid, i) < c.len) acc[0][i % AW] = fma(x[i], x[i], acc[0][i % AW]);
    } else {
        unit_wait(c);
        constexpr bool ALL = GR && GRAM == 2;  // all pairs: the rows are held together
        VB v[ALL ? KB : 1][E], vl[E];
        if constexpr (GR && GRAM == 1) lds_row<NT>(unit_row(c, d0, nd - 1) + off, vl);
#pragma unroll
        for (int r = 0; r < KB; r++) {
            if (r >= nd) break;
            VB(&vr)[E] = v[ALL ? r : 0];
            lds_row<NT>(unit_row(c, d0, r) + off, vr);
#pragma unroll
            for (int i = 0; i < E; i++) {
                if (!FULL && e0 + place<VB, E, NT>(tid, i) >= c.len) continue;
                acc[r][i % AW] = fma(x[i], vr[i], acc[r][i % AW]);
                if constexpr (GR && GRAM == 1) {
                    if (r < KB - 1 && r < nd - 1)
                        acc[KB + (r < KB - 1 ? r : 0)][i % AW] =
                            fma(vl[i], vr[i], acc[KB + (r < KB - 1 ? r : 0)][i % AW]);
                }
                if constexpr (ALL) {
#pragma unroll
                    for (int q = 0; q < r; q++)
                        acc[KB + r * (r - 1) / 2 + q][i % AW] =
                            fma(vr[i], v[q][i], acc[KB + r * (r - 1) / 2 + q][i % AW]);
                }
            }
        }
        unit_free(c);
    }
}

// One pass over the CTA's part: w -= sum of the nu rows from u0 (coefficients
// cf), store, then (FIN) the squared norm or the dots with the nd <= KB rows
// from d0 and, with GR, the rows' own inner products: GRAM 2 all pairs, GRAM 1
// the newest row (d0 + nd - 1) with the others.
template <typename VB, int KB, int NT, int GRAM, bool GR, bool FIN, int NA>
__device__ __forceinline__ void gs_pass(Ctx<VB, KB, NT> &c, const VB *src, bool from_global, VB *dst, int u0,
                                        int nu, const VB *cf, int d0, int nd, double (&out)[NA]) {
    constexpr int E = gs_elems<VB, KB, NT>(), T = gs_tile<VB, KB, NT>();
    constexpr int AW = chains<VB, KB, GRAM>();
    const int tid = threadIdx.x;
    constexpr int D = sizeof(VB) == 8 ? 3 : 2;  // tiles of w on their way (global w)
    VB acc[NA][AW], xn[D][E];
#pragma unroll
    for (int i = 0; i < NA; i++)
#pragma unroll
        for (int q = 0; q < AW; q++) acc[i][q] = VB(0);
    const int step = c.pass & 1 ? -T : T;
    int e0 = c.pass & 1 ? (c.tiles - 1) * T : 0;
    c.pass++;
    if (from_global) {
#pragma unroll
        for (int d = 0; d < D; d++)
#pragma unroll
            for (int i = 0; i < E; i++) {
                const int e = e0 + d * step + place<VB, E, NT>(tid, i);
                xn[d][i] = e >= 0 && e < c.len ? src[e] : VB(0);
            }
    }
    for (int t = 0; t < c.tiles; t++, e0 += step) {
        VB x[E];
        if (from_global) {
#pragma unroll
            for (int i = 0; i < E; i++) {
                x[i] = xn[0][i];
                const int e = e0 + D * step + place<VB, E, NT>(tid, i);
#pragma unroll
                for (int d = 0; d + 1 < D; d++) xn[d][i] = xn[d + 1][i];
                xn[D - 1][i] = e >= 0 && e < c.len ? src[e] : VB(0);
            }
        } else {
#pragma unroll
            for (int i = 0; i < E; i++) {
                const int e = e0 + place<VB, E, NT>(tid, i);
                x[i] = e < c.len ? src[e] : VB(0);
            }
        }
        if (e0 + T <= c.len) gs_tile_pass<VB, KB, NT, GRAM, GR, FIN, true>(c, e0, x, dst, u0, nu, cf, d0, nd, acc);
        else gs_tile_pass<VB, KB, NT, GRAM, GR, FIN, false>(c, e0, x, dst, u0, nu, cf, d0, nd, acc);
    }
#pragma unroll
    for (int i = 0; i < NA; i++) {
        out[i] = (double)acc[i][0];
        if constexpr (AW == 8)
#pragma unroll
            for (int q = 0; q < 4; q++) acc[i][q] += acc[i][q + 4];
        if constexpr (AW >= 4)
            out[i] = ((double)acc[i][0] + (double)acc[i][1]) + ((double)acc[i][2] + (double)acc[i][3]);
    }
}

// ---- exchange ---------------------------------------------------------------------
// Value q belongs to rank q mod cs of every cluster.  Each warp sends its sums
// to the owner in its cluster; the owner adds them and publishes the cluster's
// sum in device memory; the owners (one CTA of each cluster, so that few
// readers wait on a line) add the clusters' sums and send the total to every
// CTA of their cluster.  All sums in a fixed order.

// The warp's sums of NV values, as values q0.. of exchange seq.
template <int NV, typename VB, int KB, int NT>
__device__ __forceinline__ void publish(Ctx<VB, KB, NT> &c, double (&v)[NV], int q0, unsigned seq) {
    constexpr int NW = NT / 32;
    warp_totals<NV>(v, c.lane);
    if (c.lane % (32 / NV) == 0) {
        const int q = q0 + c.lane / (32 / NV), cs = c.a->cs;
        put_cluster(c.part + (((seq & 1) * kGsVals + (q / cs) * cs) * NW + c.rank * NW + c.wv) * 16, q % cs,
                    v[0], seq);
    }
}

// Sum of value q over the warps of the cluster (owner's warp).
template <typename VB, int KB, int NT>
__device__ __forceinline__ double cluster_sum(Ctx<VB, KB, NT> &c, int q, unsigned seq) {
    constexpr int NW = NT / 32;
    const int cs = c.a->cs, cnt = cs * NW;
    const unsigned at = c.part + (((seq & 1) * kGsVals + (q / cs) * cs) * NW) * 16;
    constexpr int SL = 8 * NW / 32;
    double r[SL];
    bool got[SL];
#pragma unroll
    for (int s = 0; s < SL; s++) {
        got[s] = s * 32 + c.lane >= cnt;
        r[s] = 0.0;
    }
    Patience w;
    for (;;) {
        bool all = true;
#pragma unroll
        for (int s = 0; s < SL; s++)
            if (!got[s]) {
                double v;
                got[s] = get_shared(at + (s * 32 + c.lane) * 16, seq, v);
                if (got[s]) r[s] = v;
                all = all && got[s];
            }
        if (__all_sync(0xffffffffu, all)) break;
        if (__any_sync(0xffffffffu, w.expired(*c.a, c.look))) {
            give_up(c);
            break;
        }
    }
    double v[1] = {r[0]};
#pragma unroll
    for (int s = 1; s < SL; s++)
        if (s * 32 < cnt) v[0] += r[s];
    warp_totals<1>(v, c.lane);
    return v[0];
}

// Sum of value q over the clusters.
template <typename VB, int KB, int NT>
__device__ __forceinline__ double grid_sum(Ctx<VB, KB, NT> &c, int q, unsigned seq) {
    constexpr int SL = kGsMaxClusters / 32;
    const int nc = gridDim.x / c.a->cs;
    const ulonglong2 *at = c.a->slots + ((size_t)(seq & 1) * kGsVals + q) * kGsMaxClusters + c.lane;
    double r[SL];
    bool got[SL];
#pragma unroll
    for (int s = 0; s < SL; s++) {
        got[s] = s * 32 + c.lane >= nc;
        r[s] = 0.0;
    }
    Patience w;
    for (;;) {
        bool all = true;
#pragma unroll
        for (int s = 0; s < SL; s++)
            if (!got[s]) {
                double v;
                got[s] = get_global(at + s * 32, seq, v);
                if (got[s]) r[s] = v;
                all = all && got[s];
            }
        if (__all_sync(0xffffffffu, all)) break;
        if (__any_sync(0xffffffffu, w.expired(*c.a, c.look))) {
            give_up(c);
            break;
        }
    }
    double v[1] = {r[0]};
#pragma unroll
    for (int s = 1; s < SL; s++)
        if (s * 32 < nc) v[0] += r[s];
    warp_totals<1>(v, c.lane);
    return v[0];
}

// The owner's share of exchange seq over nv values.
template <typename VB, int KB, int NT>
__device__ __forceinline__ void relay(Ctx<VB, KB, NT> &c, int nv, unsigned seq) {
    constexpr int NW = NT / 32;
    const int cs = c.a->cs, ci = blockIdx.x / cs;
    for (int q = c.rank + cs * c.wv; q < nv; q += cs * NW) {
        const double s = cluster_sum(c, q, seq);
        if (c.lane == 0)
            put_global(c.a->slots + ((size_t)(seq & 1) * kGsVals + q) * kGsMaxClusters + ci, s, seq);
    }
    for (int q = c.rank + cs * c.wv; q < nv; q += cs * NW) {
        const double s = grid_sum(c, q, seq);
        if (c.lane < cs) put_cluster(c.bc + ((seq & 1) * kGsVals + q) * 16, c.lane, s, seq);
    }
}

// Totals q0 .. q0 + 31 of exchange seq, one per lane (0 from nv on).
template <typename VB, int KB, int NT>
__device__ __forceinline__ double totals(Ctx<VB, KB, NT> &c, int q0, int nv, unsigned seq) {
    bool got = q0 + c.lane >= nv;
    double r = 0.0;
    Patience w;
    for (;;) {
        if (!got) {
            double v;
            got = get_shared(c.bc + ((seq & 1) * kGsVals + q0 + c.lane) * 16, seq, v);
            if (got) r = v;
        }
        if (__all_sync(0xffffffffu, got)) break;
        if (__any_sync(0xffffffffu, w.expired(*c.a, c.look))) {
            give_up(c);
            break;
        }
    }
    return r;
}

// The scalar warp of CTA 0: while the compute warps take the last update, it
// rotates the column by the earlier Givens rotations; then it sums the norm
// over the clusters and ends the step.  The roots, and then the quotients, are
// taken by different lanes in one instruction sequence each: an FP64 sequence
// takes as long for one lane as for 32.
template <typename VB, int KB, int NT>
__device__ void scalar_warp(Ctx<VB, KB, NT> &c, unsigned seq, bool raw) {
    const GsArgs<VB> &a = *c.a;
    const xb::GmDev &st = a.st;
    const double *h = c.S->hcol;
    const int j = a.j, lane = c.lane;
    double len2 = 0.0, t = 0.0, gj = 0.0, rg = 0.0, tau = 0.0;
    if (raw) {
        for (int i = lane; i <= j; i += 32) a.col[i] = h[i];
    } else {
        gj = st.g[j];
        rg = fabs(gj) / st.misc[xb::GM_BNORM];
        tau = st.misc[xb::GM_TAU];
        for (int i = lane; i <= j; i += 32) len2 = fma(h[i], h[i], len2);
        len2 = xbd::warp_sum(len2);
        t = h[0];
        for (int i = 0; i < j; i++) {
            const double cs = __ldg(st.cs + i), sn = __ldg(st.sn + i), b = h[i + 1];
            if (lane == 0) a.col[i] = cs * t + sn * b;
            t = -sn * t + cs * b;
        }
    }
    const double nn = grid_sum(c, 0, seq);
    if (!c.fine) return;
    if (raw) {
        if (lane == 0) a.col[j + 1] = sqrt(nn);
        return;
    }
    const double rr2 = fma(t, t, nn);
    double hn, rr;
    if (rr2 > 1e-280 && rr2 < 1e280) {
        const double q = sqrt(lane == 0 ? nn : rr2);
        hn = __shfl_sync(0xffffffffu, q, 0);
        rr = __shfl_sync(0xffffffffu, q, 1);
    } else {
        hn = sqrt(nn);
        rr = hypot(t, hn);
    }
    // one word tells the host: no copy in the stream, no fence
    auto tell = [&](int stop) {
        if (stop) st.misc[xb::GM_STOP] = (double)stop;
        *reinterpret_cast<volatile unsigned long long *>(a.late + (a.tag & 1)) = 4 * a.tag + stop;
    };
    const double q = (lane == 0 ? t : lane == 1 ? hn : 1.0) / (lane < 2 ? rr : hn);
    const double cs = __shfl_sync(0xffffffffu, q, 0), sn = __shfl_sync(0xffffffffu, q, 1);
    const double inv = __shfl_sync(0xffffffffu, q, 2);
    if (lane != 0) return;
    st.misc[xb::GM_LEN2] = len2;
    if (rr == 0.0) {  // A v_j lies in span(v_0..v_{j-1}) with a zero pivot: singular
        a.col[j] = t;
        a.col[j + 1] = hn;
        tell(2);
        return;
    }
    st.cs[j] = cs;
    st.sn[j] = sn;
    a.col[j] = rr;
    a.col[j + 1] = 0.0;
    st.g[j + 1] = -sn * gj;
    st.g[j] = cs * gj;
    const double res = sn * rg;
    st.misc[xb::GM_RES] = res;
    st.misc[xb::GM_K] = (double)(j + 1);
    if (hn <= 1e-14 * sqrt(len2 + hn * hn)) {  // happy breakdown: the Krylov space is invariant
        st.sc[j + 1] = 0.0;
        st.scf[j + 1] = 0.0f;
        tell(1);
        return;
    }
    st.sc[j + 1] = inv;
    st.scf[j + 1] = (float)inv;
    tell(res <= tau ? 1 : 0);
}

// What bounds it and why this form.  At small n the time of an
// orthogonalisation is that of its chain of inner products; at large n it is
// the FP64 pipe (two FMAs per basis element) or, for the FP32 basis, HBM.  So:
// one launch; few warps (a sum over the threads of an SM costs FP64 time in
// proportion to their number); w read once and written once; and an exchange
// per block of KB rows.  For MGS that is the same method in exact arithmetic:
//   (w - sum_{k<i} c_k V_k, V_i) = (w, V_i) - sum_{k<i} c_k (V_k, V_i),
// with k over the earlier rows of the block, so the dots of a block are all
// taken with the same w and corrected by the rows' own inner products.  In
// rounding, c_i carries eps ||w|| of the block's first w, not of what the earlier
// rows left: as much as w's own updates carry into the result, so the loss against
// the rows as a whole is MGS's (w = 1e4 V_0 + u: ||w'|| off by 1.4e-12, 0.9e-12 one at
// a time; against the block's later rows 1e-13, 1e-17 one at a time).  In
// GMRES (GRAM 1) the products are kept from the step in which a row was the newest
// (at most KB - 1 more dots a step); a sweep against rows it has not seen
// (GRAM 2) takes them in the same pass.
//
// Measured (GB300, launch included; the launch per row or per 4-8 rows it
// replaced in brackets): FP64 MGS against 20 rows of n = 103,071 49 us (225);
// DGKS against 40 rows of n = 2.1M 614 us (940; the FP64 pipe's floor 557); BCGS
// against 30 rows of n = 16.8M 2.12 ms (2.28; floor 1.68); MGS against 12 rows
// of n = 16.8M 953 us (1090); FP32 BCGS against 16 rows of n = 2.1M 58 us.
template <typename VB, int KB, int NT, int GRAM, bool SM>
__global__ void __launch_bounds__(NT + 64, 1) k_gs(const __grid_constant__ GsArgs<VB> a) {
    if (a.st.misc && a.st.misc[xb::GM_STOP] != 0.0) return;
    if (cluster_size() != a.cs) {  // launched in another shape (a tool's replay): no peers to talk to
        if (threadIdx.x == 0) *reinterpret_cast<volatile int *>(a.err) = 1;
        return;
    }
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ GsShared<VB, KB, NT> S;
    constexpr int NG = gram_count(KB, GRAM), NW = NT / 32;
    constexpr int NX = KB + NG <= 1 ? 1 : KB + NG <= 2 ? 2 : KB + NG <= 4 ? 4 : KB + NG <= 8 ? 8 : 16;
    const int tid = threadIdx.x;
    const bool raw = !a.st.misc || a.st.misc[xb::GM_RAW] != 0.0;
    const int k = a.j + 1;
    const int64_t c0 = blockIdx.x * a.chunk;
    Ctx<VB, KB, NT> c;
    c.S = &S;
    c.a = &a;
    c.Vc = a.V + c0;
    c.part = sptr(dyn);
    c.bc = c.part + 2 * kGsVals * NW * 16;
    c.ring = c.bc + 2 * kGsVals * 16;
    c.len = (int)max((int64_t)0, min(a.chunk, a.n - c0));
    c.tiles = (c.len + gs_tile<VB, KB, NT>() - 1) / gs_tile<VB, KB, NT>();
    c.rank = cluster_rank();
    c.lane = tid & 31;
    c.wv = tid >> 5;
    c.row0 = (unsigned)(uintptr_t)c.Vc;
    c.pitch = (unsigned)(a.ld * sizeof(VB));
    c.look = a.look;
    c.st = c.ph = c.pass = 0;
    c.fine = true;
    for (int i = tid; i < gs_xch_bytes<NT>() / 16; i += NT + 64)
        reinterpret_cast<ulonglong2 *>(dyn)[i] = make_ulonglong2(0, 0);
    if (tid == 0) {
        S.abort = 0;
        for (int s = 0; s < a.stages; s++) {
            mbar_init(sptr(&S.full[s]), 1);
            mbar_init(sptr(&S.empty[s]), NW);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cluster_sync();
    unsigned seq = a.base;
    constexpr bool either = GRAM == 0 && sizeof(VB) == 8;
    const bool blocks = either ? a.method == XB_ORTHO_MGS || a.method == XB_ORTHO_BCGS : GRAM != kCgs;
    const int nb = (k + KB - 1) / KB, rounds = a.method == XB_ORTHO_DGKS ? 2 : 1;
    const int groups = (k + kGsVals - 1) / kGsVals;
    if (c.wv == NW) {  // producer: the units in the order the passes take them
        // a pass's pending rows are read for the last time: their lines make way
        // in L2 for the rows that the next pass reads again
        uint64_t keep, last;
        asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(keep));
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(last));
        int pass = 0;
        if (blocks) {
            for (int b = 0; b <= nb; b++, pass++)
                for (int i = 0; i < c.tiles; i++) {
                    const int t = pass & 1 ? c.tiles - 1 - i : i;
                    if (b > 0) produce(c, t, (b - 1) * KB, min(KB, k - (b - 1) * KB), last);
                    if (b < nb) produce(c, t, b * KB, min(KB, k - b * KB), keep);
                }
        } else {
            for (int r = 0; r <= rounds; r++)
                for (int d0 = 0; d0 < k; d0 += KB, pass++) {
                    if (r == rounds && d0 > 0) break;  // last: the update alone
                    for (int i = 0; i < c.tiles; i++) {
                        const int t = pass & 1 ? c.tiles - 1 - i : i;
                        if (r > 0 && d0 == 0)
                            for (int i0 = 0; i0 < k; i0 += KB) produce(c, t, i0, min(KB, k - i0), keep);
                        if (r < rounds) produce(c, t, d0, min(KB, k - d0), keep);
                    }
                }
        }
    } else if (c.wv > NW) {
        if (blockIdx.x == 0) {
            bar_sync(2, NT + 32);
            if (!*reinterpret_cast<volatile int *>(&S.abort))
                scalar_warp(c, seq + (blocks ? nb : rounds * groups) + 1, raw);
        }
    } else {
        VB *wg = a.w + c0;
        VB *wl = SM ? reinterpret_cast<VB *>(dyn + gs_xch_bytes<NT>() + (size_t)a.stages * KB * gs_pitch<VB, KB, NT>())
                    : wg;
        const VB *src = wg;
        bool fg = true;                // w comes from global memory
        VB *dst = SM ? wl : nullptr;   // the first pass brings it in
        int u0 = 0, nu = 0;
        const VB *cu = S.cf;
        if (blocks) {
            cu = S.cfw[c.wv];
            for (int b = 0; b < nb && c.fine; b++) {
                const int d0 = b * KB, nd = min(KB, k - d0);
                const bool last = b == nb - 1;
                double s1 = 0.0, g[KB];
#pragma unroll
                for (int i = 0; i < KB; i++) g[i] = 0.0;
                if (c.lane < nd) {
                    s1 = a.st.sc ? a.st.sc[d0 + c.lane] : 1.0;
                    if constexpr (GRAM == 1) {
                        if (!(last && c.lane == nd - 1))
#pragma unroll
                            for (int i = 0; i < KB - 1; i++)
                                if (i < c.lane) g[i] = a.st.gram[(size_t)(d0 + c.lane) * 8 + i];
                    }
                }
                seq++;
                const bool gr = GRAM == 2 || (GRAM == 1 && last);
                int nv = nd;
                if constexpr (GRAM != 0) {
                    if (gr) {
                        double v[NX], o[KB + NG];
                        nv = KB + NG;
                        gs_pass<VB, KB, NT, GRAM, true, false>(c, src, fg, dst, u0, nu, cu, d0, nd, o);
#pragma unroll
                        for (int i = 0; i < NX; i++) v[i] = i < KB + NG ? o[i] : 0.0;
                        publish<NX>(c, v, 0, seq);
                    }
                }
                if (GRAM != 2 && !gr) {
                    double v[KB];
                    gs_pass<VB, KB, NT, GRAM, false, false>(c, src, fg, dst, u0, nu, cu, d0, nd, v);
                    publish<KB>(c, v, 0, seq);
                }
                relay(c, nv, seq);
                const double tot = totals(c, 0, nv, seq);
                if (__any_sync(0xffffffffu, !c.fine || *reinterpret_cast<volatile int *>(&S.abort))) {
                    c.fine = false;
                    break;
                }
                // lane i: t = (V_i, w) as MGS finds it, u = the coefficient of V_i
                const double s2 = s1 * s1;
                double t = c.lane < nd ? tot : 0.0;
                if constexpr (GRAM == 2) {
#pragma unroll
                    for (int i = 0; i < KB - 1; i++) {
                        const double x =
                            __shfl_sync(0xffffffffu, tot, min(31, KB + c.lane * (c.lane - 1) / 2 + i));
                        if (i < c.lane && c.lane < nd) g[i] = x;
                    }
                } else if constexpr (GRAM == 1) {
                    if (last) {
#pragma unroll
                        for (int i = 0; i < KB - 1; i++) {
                            const double x = __shfl_sync(0xffffffffu, tot, KB + i);
                            if (c.lane == nd - 1 && i < c.lane) g[i] = x;
                        }
                        if (blockIdx.x == 0 && c.wv == 0 && c.lane >= KB && c.lane < KB + nd - 1)
                            a.st.gram[(size_t)(d0 + nd - 1) * 8 + c.lane - KB] = tot;
                    }
                }
                double u = s2 * t;
                if constexpr (GRAM != 0) {
                    // a row that w is orthogonal to takes nothing away, whatever its
                    // products: they overflow sooner than one row's dot does.  Looked at
                    // only where a total is not finite (in every block it cost 0.25 us), and
                    // not in GMRES, whose rows' norms are finite squares
                    auto correct = [&](bool look) {
#pragma unroll
                        for (int i = 0; i < KB - 1; i++) {
                            const double ci = __shfl_sync(0xffffffffu, u, i);
                            if (c.lane > i && c.lane < nd && !(look && ci == 0.0)) {
                                t = fma(-ci, g[i], t);
                                u = s2 * t;
                            }
                        }
                    };
                    if (GRAM == 2 && __any_sync(0xffffffffu, (__double2hiint(tot) & 0x7ff00000) == 0x7ff00000))
                        correct(true);
                    else
                        correct(false);
                }
                if (c.lane < KB) S.cfw[c.wv][c.lane] = (VB)u;
                if (c.wv == 0 && c.lane < nd) S.hcol[d0 + c.lane] = s1 * t;
                __syncwarp();
                u0 = d0;
                nu = nd;
                src = dst = wl;
                fg = !SM;
            }
        } else if constexpr (either || GRAM == kCgs) {
            for (int r = 0; r < rounds && c.fine; r++)
                for (int g0 = 0; g0 < k && c.fine; g0 += kGsVals) {
                    const int kg = min(kGsVals, k - g0);
                    seq++;
                    for (int d0 = g0; d0 < g0 + kg; d0 += KB) {
                        double v[KB];
                        gs_pass<VB, KB, NT, 0, false, false>(c, src, fg, dst, 0, r > 0 && d0 == 0 ? k : 0, cu, d0,
                                                         min(KB, k - d0), v);
                        publish<KB>(c, v, d0 - g0, seq);
                        src = wl;
                        fg = !SM;
                        // stored again by the next update
                        dst = r + 1 < rounds && d0 + KB >= k ? wl : nullptr;
                    }
                    relay(c, kg, seq);
                    if (c.wv == 0)
                        for (int q0 = 0; q0 < kg; q0 += 32) {
                            const double tot = totals(c, q0, kg, seq);
                            const int i = g0 + q0 + c.lane;
                            if (q0 + c.lane < kg) {
                                const double s1 = a.st.sc ? a.st.sc[i] : 1.0, h = s1 * tot;
                                S.hcol[i] = r > 0 ? S.hcol[i] + h : h;
                                S.cf[i] = (VB)(s1 * h);
                            }
                        }
                    if (bar_any(1, NT, !c.fine)) c.fine = false;
                }
            nu = k;
        }
        if (blockIdx.x == 0) bar_arrive(2, NT + 32);
        if (c.fine) {
            double v[1];
            gs_pass<VB, KB, NT, GRAM, false, true>(c, src, fg, wg, u0, nu, cu, 0, 0, v);
            publish<1>(c, v, 0, seq + 1);
            if (c.rank == 0 && c.wv == 0) {
                const double s = cluster_sum(c, 0, seq + 1);
                if (c.lane == 0)
                    put_global(a.slots + (size_t)((seq + 1) & 1) * kGsVals * kGsMaxClusters + blockIdx.x / a.cs, s,
                               seq + 1);
            }
        }
    }
    // no CTA leaves while another of its cluster may write to its slots, or before
    // its own copies
    __syncwarp();
    cluster_sync();
    if (c.wv == NW && *reinterpret_cast<volatile int *>(&S.abort)) drain(c);
}

// Largest number of clusters of cs CTAs, one CTA per SM, that the GPU holds.
template <typename K>
int max_clusters(K kernel, int threads, int cs, int *clusters) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = xb::kGsDynMax;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nc = 0;
    XB_CUDA(cudaOccupancyMaxActiveClusters(&nc, kernel, &cfg));
    *clusters = std::min(nc, kGsMaxClusters);
    return XB_OK;
}

template <typename VB, int KB, int NT, int GRAM, bool SM>
int launch(GsArgs<VB> &a, int clusters, size_t smem, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * a.cs));
    cfg.blockDim = dim3(NT + 64);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = a.cs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeCooperative;
    at[1].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    XB_CUDA(cudaLaunchKernelEx(&cfg, k_gs<VB, KB, NT, GRAM, SM>, a));
    return XB_OK;
}

// The numbers of a launch of `used` exchanges, after those of the launch before.
// They never pass 0: before they would, the grid's slots, in which a number may
// have stood since the last time round, are cleared and the count begins again
// (a launch clears its CTAs' slots itself).
int gs_numbers(xb_plan *p, unsigned used, unsigned *base, cudaStream_t s) {
    const bool pass = p->gs_number > 0xffffffffu - used;
    if (pass || p->gs_recount) XB_CUDA(cudaMemsetAsync(p->d_ticket + kGsSlotsAt, 0, kGsSlotBytes, s));
    if (pass) p->gs_number = 0;
    p->gs_recount = false;
    *base = p->gs_number;
    p->gs_number += used;
    return XB_OK;
}

template <typename VB, int KB, int GRAM, int NT = 256>
int plan_launch(xb_plan *p, GsArgs<VB> &a, cudaStream_t s) {
    struct Limits {
        int nc[9];
    };
    static xb::PerDevice<Limits> limits;
    Limits lim;
    int dev = 0;
    XB_CUDA(cudaGetDevice(&dev));
    XB_TRY(limits.get(dev, [](Limits &l) {
        XB_CUDA(cudaFuncSetAttribute(k_gs<VB, KB, NT, GRAM, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     xb::kGsDynMax));
        XB_CUDA(cudaFuncSetAttribute(k_gs<VB, KB, NT, GRAM, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     xb::kGsDynMax));
        for (int cs : {2, 4, 8})
            XB_TRY(max_clusters(k_gs<VB, KB, NT, GRAM, true>, NT + 64, cs, &l.nc[cs]));
        return (int)XB_OK;
    }, &lim));
    // Larger clusters make the exchange cheaper (3.1 / 3.5 / 4.6 us with 8 / 4 / 2
    // CTAs) but leave SMs out (120 / 144 / 152 of 152 hold a CTA).  DGKS against 20
    // rows, clusters of 2 / 4 / 8: n = 27,000 32.0 / 30.7 / 30.6 us; against 16
    // rows, n = 262,144 53.7 / 54.9 / 60.9 us (BCGS 44.5 / 42.0 / 44.7); n = 1M
    // 191 / 201 / 237 us.
    a.cs = a.n < 150000 ? 8 : (a.n < 400000 ? 4 : 2);
    if (p->gs_ctas)
        while (a.cs > 2 && a.cs > p->gs_ctas) a.cs /= 2;
    if (lim.nc[a.cs] < 1) return xb::set_error(XB_ECUDA, "orthogonalisation: no cluster of %d fits", a.cs);
    // a CTA has at least an element per thread (n = 9,600, MGS against 20 rows:
    // 33.0 us with 256 elements a CTA, 42.9 with 1024)
    const int64_t per = NT;
    const int64_t want = (a.n + per * a.cs - 1) / (per * a.cs);
    const int most = p->gs_ctas ? std::min(lim.nc[a.cs], p->gs_ctas / a.cs) : lim.nc[a.cs];
    const int nc = (int)std::max<int64_t>(1, std::min<int64_t>(most, want));
    const int64_t G = (int64_t)nc * a.cs;
    a.chunk = ((a.n + G - 1) / G + 3) / 4 * 4;
    // w in shared memory when three stages fit beside it
    const size_t stage = (size_t)KB * gs_pitch<VB, KB, NT>(), fixed = gs_xch_bytes<NT>();
    const size_t wb = (size_t)a.chunk * sizeof(VB);
    const bool sm = fixed + 3 * stage + wb <= (size_t)xb::kGsDynMax;
    p->gs_kb = KB;
    p->gs_held = sm;
    a.stages = (int)std::min<size_t>(kGsMaxStages, (xb::kGsDynMax - fixed - (sm ? wb : 0)) / stage);
    const size_t smem = fixed + a.stages * stage + (sm ? wb : 0);
    const int k = a.j + 1;
    const bool blocks = a.method == XB_ORTHO_MGS || a.method == XB_ORTHO_BCGS;
    const int sums = blocks ? (k + KB - 1) / KB
                            : (a.method == XB_ORTHO_DGKS ? 2 : 1) * ((k + kGsVals - 1) / kGsVals);
    XB_TRY(gs_numbers(p, (unsigned)sums + 1, &a.base, s));
    return sm ? launch<VB, KB, NT, GRAM, true>(a, nc, smem, s) : launch<VB, KB, NT, GRAM, false>(a, nc, smem, s);
}

template <typename VB>
int gs_run(xb_plan *p, GsArgs<VB> &a, bool seen, cudaStream_t s) {
    a.stop = p->d_ticket + 64;
    a.polls = p->gs_polls;
    a.look = a.polls ? a.polls : 256u;
    a.slots = reinterpret_cast<ulonglong2 *>(p->d_ticket + kGsSlotsAt);
    a.err = reinterpret_cast<int *>(p->h_pin + 60);
    a.late = reinterpret_cast<unsigned long long *>(p->h_pin + 40);
    a.tag = ++p->gs_tag;
    // Rows of a block, and threads.  Long vectors want few rows: MGS pays for the
    // products of its blocks (GMRES(10) of n = 8M, us a step: blocks of 8 510, of 4
    // 474, of 2 422; n = 2.1M, GMRES(20): 191, 202, 197), and a unit of fewer rows
    // than the block has leaves undone the copies that hide the latency (against 1
    // row of n = 16.8M, blocks of 8 / 2: DGKS 484 / 285 us; 4 rows, 8 / 4: 680 / 604).
    // Without products in the way 512 threads go with it (256 / 512: DGKS against 3,
    // 9 rows 558 / 483, 1416 / 1329; BCGS against 5 513 / 387).  An FP32 basis of n =
    // 2.1M / 16.8M, GMRES(10): MGS in 8 90 / 455, in 4 84 / 441; DGKS 108 / 574, 95 / 546
    // (n = 1M, GMRES(30): MGS 74, 76).  MGS has one block size for a whole solve (st.gram).
    const bool longv = a.n >= 3000000;
    const int k = a.j + 1;
    if constexpr (sizeof(VB) == 8) {
        if (longv && (a.method != XB_ORTHO_MGS || k == 1)) {
            // (MGS against one row has no products)
            if (k <= 2) return plan_launch<VB, 2, 0, 512>(p, a, s);
            if (k <= 4 || a.method == XB_ORTHO_BCGS) return plan_launch<VB, 4, 0, 512>(p, a, s);
            return plan_launch<VB, 8, 0, 512>(p, a, s);
        }
    } else {
        if (a.n >= 1500000 && a.method != XB_ORTHO_BCGS)
            return a.method == XB_ORTHO_MGS ? plan_launch<VB, 4, 1>(p, a, s) : plan_launch<VB, 4, kCgs>(p, a, s);
    }
    if (a.method == XB_ORTHO_BCGS) return plan_launch<VB, 4, 0>(p, a, s);
    if (a.method != XB_ORTHO_MGS) return plan_launch<VB, 8, sizeof(VB) == 8 ? 0 : kCgs>(p, a, s);
    if constexpr (sizeof(VB) == 8) {
        if (seen && longv) return plan_launch<VB, 2, 1>(p, a, s);
        if (!seen) {
            // n = 262,144 (16 rows): blocks of 4 / 2 59.9 / 61.5 us; n = 1M (20
            // rows) 162 / 151 us: beyond, the rows' own products cost more FP64
            // time than the exchanges they save
            if (a.n < 600000) return plan_launch<VB, 4, 2>(p, a, s);
            return plan_launch<VB, 2, 2>(p, a, s);
        }
    }
    return plan_launch<VB, 8, 1>(p, a, s);
}

}  // namespace

namespace xb {

size_t gs_scratch_bytes() { return kGsSlotsAt * sizeof(unsigned) + kGsSlotBytes; }

int gs_check(xb_plan *p, cudaStream_t s) {
    volatile int *err = reinterpret_cast<volatile int *>(p->h_pin + 60);
    if (!*err) return XB_OK;
    *err = 0;
    XB_CUDA(cudaMemsetAsync(p->d_ticket + 64, 0, sizeof(unsigned), s));
    XB_CUDA(cudaStreamSynchronize(s));  // the next launch may be on another stream
    return set_error(XB_ETIMEOUT, "orthogonalisation: a grid exchange ran out of time");
}

template <typename VB>
int gm_ortho_step(xb_plan *p, GmDev st, int64_t n, const VB *V, int64_t ld, VB *w, int j, int ortho,
                  bool seen, cudaStream_t s) {
    GsArgs<VB> a{};
    a.n = n;
    a.ld = ld;
    a.V = V;
    a.w = w;
    a.st = st;
    a.col = st.H + (size_t)j * (st.M + 1);
    a.j = j;
    a.method = ortho;
    return gs_run<VB>(p, a, seen, s);
}
template int gm_ortho_step<double>(xb_plan *, GmDev, int64_t, const double *, int64_t, double *, int,
                                   int, bool, cudaStream_t);
template int gm_ortho_step<float>(xb_plan *, GmDev, int64_t, const float *, int64_t, float *, int, int,
                                  bool, cudaStream_t);

int ortho_sweep(xb_plan *p, int64_t n, int k, const double *V, int64_t ld, double *w, double *h,
                int ortho, cudaStream_t s) {
    GsArgs<double> a{};
    a.n = n;
    a.ld = ld;
    a.V = V;
    a.w = w;
    a.col = h;
    a.j = k - 1;
    a.method = ortho;
    return gs_run<double>(p, a, false, s);
}

}  // namespace xb

extern "C" int xb_orth_config(xb_plan *p, int32_t what, int64_t value) {
    if (p && what == XB_ORTH_NUMBER && value >= 0 && value <= 0xffffffffLL) {
        p->gs_recount = p->gs_recount || (unsigned)value < p->gs_number;
        p->gs_number = (unsigned)value;
        return XB_OK;
    }
    if (p && what == XB_ORTH_POLLS && value >= 0 && value <= 0x7fffffffLL) {
        p->gs_polls = (unsigned)value;
        return XB_OK;
    }
    if (p && what == XB_ORTH_CTAS && (value == 0 || (value >= 2 && value <= 0x7fffffffLL))) {
        p->gs_ctas = (int)value;
        return XB_OK;
    }
    return xb::set_error(XB_EINVAL, "orth_config: plan %p control %d value %lld", (void *)p, what, (long long)value);
}
