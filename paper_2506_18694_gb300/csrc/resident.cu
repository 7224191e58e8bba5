// A whole multigrid cycle, or the whole HSS loop of a preconditioner application, of a small 2D
// problem in ONE launch: one thread-block cluster per problem, every level in distributed shared
// memory.
//
// Why.  On grids of a few hundred nodes per side a V(2,2) cycle as separate kernels is a chain
// of 2L - 1 launches of 3-10 us each, bound by launch and tile latency, not by work.  Here a
// pass over a level is a loop over shared memory and its end a halo exchange.  Measured (GB300, us
// per V-cycle of the HSS loop, 4 levels; separate kernels / resident): complex64 17^2 35 / 10, 65^2
// 36 / 15.6, 129^2 32 / 19, 257^2 35 / 30; complex128 33^2 136 / 35, 65^2 136 / 55.  A pass is bound by
// the latency of one dependent chain of about 330 cycles, plus about 500 for an exchange.
//
// Layout.  CTA r of the cluster owns rows f(r) .. f(r + 1) - 1 of level 0, f(r) = floor(r nn / cs),
// and on level l + 1 the rows J whose fine row 2J it owns, so that restriction and prolongation
// touch only its own rows and one halo row on each side.  Levels from `dist` on are small: every
// CTA holds all of them and runs them redundantly, with block barriers only.  A level keeps two
// iterates A and B (even row pitch, zero columns beside the row for the missing neighbours of both
// sides; one halo row above and below) and its right side.  A pass reads one iterate, writes the
// other, and sends its first and last rows to the halo rows of the neighbouring CTAs.
//
// Synchronisation.  Halo rows travel as st.async, which count their bytes on a memory barrier of
// the receiver: the pass ends when the block's threads are done and both halo rows are there (one
// remote-store latency, about 500 cycles; remote stores and a cluster barrier take about 760, a
// fence and a remote arrival 1600).  Two barriers per
// direction alternate, so that a neighbour one pass ahead never counts on the running one; it is
// at most one pass ahead, because it needs our rows, and each of our threads that reads a halo row
// sends its result to the same neighbour after that read.  The right side of the first replicated
// level goes to every CTA by bulk copies; a split cluster barrier (arrive after the replicated
// levels, wait before the next right side's first store) keeps a CTA from overwriting rows that a
// copy to a CTA far away may still be reading, and its copies from overwriting one in use: halo
// exchanges hold back adjacent CTAs only, a CTA six rows of them away can be a step behind.
//
// Every wait is bounded (spin_limit polls): a CTA that gives up skips the rest of its passes, but not
// the cluster barriers; its neighbours' waits run out in turn, and the launch ends with the status
// recorded and a result of NaN.  That a wait ran out is read by every thread behind the pass's block barrier,
// from a word that is not written again before the next one, so the whole CTA gives up at the same pass
// (a barrier that carries it itself, __syncthreads_or, made a cycle 1 to 3 % slower).  What others
// sent to a CTA that gave up is still on its way when the passes end: the CTAs of such a cluster tell
// one another how many passes and copies they sent, and each waits for its own (give_up).
//
// Work split of a pass: complex64, a thread takes two neighbouring columns (one 16-byte and two
// 8-byte shared loads per row) and 1, 2 or 4 rows; complex128, two lanes take the real and the
// imaginary part of one node and exchange the sums they need (the FP64 pipe takes 64 cycles per
// warp instruction whatever the number of active lanes, so a pass costs what its longest lane
// executes).  Boundary nodes, with their class weights, are taken by warps of their own, so no
// warp runs both formulas.  A pass over a small level is one chain of dependent instructions, so
// what does not change between passes (which nodes a thread takes, where they lie, their class,
// whether they are sent) is worked out once and read back as one word per item.
//
// Every node's arithmetic is that of the one-pass kernels (stencil_node2, prolong_rows, rr_tile),
// so the result equals theirs bit for bit.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "internal.h"
#include "march2_common.cuh"

namespace cg = cooperative_groups;

namespace hh {

namespace {

constexpr int kResThreads = 640;
constexpr size_t kResSmemMax = 226 * 1024;

// One level as the passes of a CTA see it: R rows of its own, Ru rows the CTA above.  A, B, b:
// offsets in shared memory (entries); A, B hold the halo row above first, b the first own row,
// column i at index i + 1 of a row.  rep: every CTA holds the level whole; up, dn: a neighbour CTA
// holds rows above / below.  Work items (words in shared memory, from offset t0, r0, p0): tiles of
// a pass (tr rows each), restricted nodes of this level (from the finer one), cells that the
// prolongation to this level fills.
struct alignas(16) Lev {
    int nn, W, R, Ru;
    int A, B, b, rep;
    int up, dn, tr, tiles;
    int t0, r0, p0, restricted;
    int cells, row0, bulk0, bulkn;  // row0: first own row; bulk*: rows sent to every CTA
};

// Item words.  A tile: its first node's offset in an iterate and flags.
constexpr unsigned kOff = 0xffffu;
constexpr unsigned kTwo = 1u << 19;    // both columns of the pair are inner (rows: bits 16..18)
constexpr unsigned kUp = 1u << 20;     // its first row is the CTA's first, and is sent up
constexpr unsigned kDn = 1u << 21;     // its last row is the CTA's last, and is sent down
constexpr unsigned kVoid = 1u << 26;   // a Dirichlet node: only sent, as 0
constexpr unsigned kValid = 1u << 27;
__device__ __forceinline__ int rows_of(unsigned d) { return (d >> 16) & 7; }
__device__ __forceinline__ int kind_of(unsigned d) { return (d >> 22) & 15; }  // 8 inner, else boundary class

enum { P_SWEEP = 0, P_RESID = 1, P_HSS = 2, P_FIRST = 3 };  // P_FIRST: the first sweep from 0

// Start of the dynamic shared memory: coefficients of the levels and of the HSS step (index
// levels), the levels, the halo barriers [from above, from below][alternating] and those of the
// replicated right side [alternating], whether a wait of a halo exchange [alternating] or of the right
// side [2] ran out; for a cluster in which one did: that it did, the passes and right sides this CTA
// sent, and the bytes of a halo row of its last pass.  Then the level vectors (at kHead<T> bytes).
template <typename T> struct Head {
    PCoef<T> coef[kResMaxLevels + 1];
    Lev lv[kResMaxLevels];
    unsigned long long mb[2][2];
    unsigned long long mbr[2];
    int gave_up[3], any, rounds, copies, row_bytes;
};
template <typename T> constexpr size_t kHead = (sizeof(Head<T>) + 127) / 128 * 128;

extern __shared__ __align__(128) unsigned char res_smem[];
template <typename T>
__device__ __forceinline__ Head<T>& head() {
    return *reinterpret_cast<Head<T>*>(res_smem);
}
template <typename T>
__device__ __forceinline__ vec2<T>* vecs() {
    return reinterpret_cast<vec2<T>*>(res_smem + kHead<T>);
}

__device__ __forceinline__ unsigned saddr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned remote(unsigned a, int rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
// stores to another CTA's shared memory that count their bytes on its barrier
__device__ __forceinline__ void send(unsigned dst, Cx<float> v, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(dst),
                 "f"(v.re), "f"(v.im), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void send(unsigned dst, Cx<double> v, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(dst),
                 "d"(v.re), "d"(v.im), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void send2(unsigned dst, Cx<float> a, Cx<float> b, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst),
                 "f"(a.re), "f"(a.im), "f"(b.re), "f"(b.im), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bar_expect(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_try(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// The cluster as a CTA sees it: Dirichlet sides (bit s: side s), the level vectors' address in the
// CTAs above and below, and the number of passes that exchanged halo rows, with kDead set when a wait
// of this CTA ran out: its later passes do nothing.
constexpr int kDead = 1 << 30;
struct Res {
    int rank, cs, dir;
    unsigned base_up, base_dn, mb_up, mb_dn;  // (mb_*: the neighbour's barrier of what we send)
    int round;
    unsigned long long spin;
    __device__ __forceinline__ bool dead() const { return round & kDead; }
};

// Where a pass sends its first and last row: the addresses that, with the node's own offset in the
// iterate added, give its place in the halo row of the neighbour's iterate at offset `buf`.
struct Push {
    unsigned up, dn, bup, bdn;
};
template <typename T>
__device__ __forceinline__ Push push_rows(const Res& S, const Lev& L, int buf) {
    const unsigned e = sizeof(vec2<T>), k = (S.round & 1) * 8;
    return Push{S.base_up + (buf + L.Ru * L.W) * e, S.base_dn + (buf - L.R * L.W) * e, S.mb_up + k, S.mb_dn + k};
}

// Wait for a barrier's phase, at most `spin` polls; false when they run out.
__device__ __forceinline__ bool bounded_wait(unsigned long long* bar, unsigned parity, unsigned long long spin) {
    unsigned long long k = 0;
    while (!bar_try(saddr(bar), parity))
        if (++k > spin) return false;
    return true;
}

// End of a pass whose first and last rows were sent: thread 0 waits for the row from above, thread
// 32 for the one from below, then the block meets and sees whether a wait ran out.  The next pass that
// writes the same word comes after one more block barrier.  (pass_begin: what the pass expects.)
template <typename T>
__device__ __forceinline__ void pass_begin(const Res& S, const Lev& L) {
    Head<T>& hd = head<T>();
    const unsigned bytes = L.nn * sizeof(vec2<T>);
    if (threadIdx.x == 0 && L.up) bar_expect(saddr(&hd.mb[0][S.round & 1]), bytes);
    if (threadIdx.x == 32 && L.dn) bar_expect(saddr(&hd.mb[1][S.round & 1]), bytes);
}
template <typename T>
__device__ __forceinline__ void pass_end(Res& S, const Lev& L) {
    Head<T>& hd = head<T>();
    const int k = S.round & 1, d = threadIdx.x == 0 ? 0 : 1;
    if ((threadIdx.x == 0 && L.up) || (threadIdx.x == 32 && L.dn)) {
        if (!bounded_wait(&hd.mb[d][k], (S.round >> 1) & 1, S.spin)) {
            hd.gave_up[k] = kDead;
            hd.row_bytes = L.nn * (int)sizeof(vec2<T>);
        }
    }
    __syncthreads();
    S.round = (S.round + 1) | hd.gave_up[k];
}

__device__ __forceinline__ void st_pair(float2* p, Cx<float> a, Cx<float> b) {
    *reinterpret_cast<float4*>(p) = make_float4(a.re, a.im, b.re, b.im);
}

// Weights of an item: its neighbour groups' and omega D^{-1} (inner: centre, edges, diagonals; a
// boundary class: centre, x, y, diagonal neighbours), and the HSS step's scalars.
template <typename T> struct Wt {
    Cx<T> w[4], dinv, alpha, beta;
};
template <typename T, int MODE>
__device__ __forceinline__ Wt<T> weights(const PCoef<T>& c, int kind) {
    Wt<T> k;
    if (kind == 8) {
        for (int q = 0; q < 3; ++q) k.w[q] = c.iw[q];
        k.w[3] = cx<T>(0, 0);
        k.dinv = c.wdinv;
    } else {
        for (int q = 0; q < 4; ++q) k.w[q] = c.bw[kind][q];
        k.dinv = c.bdinv[kind];
    }
    if (MODE == P_HSS) {
        k.alpha = c.alpha;
        k.beta = c.beta;
    }
    return k;
}

// the update of one node from its stencil product ax
template <typename T, int MODE>
__device__ __forceinline__ Cx<T> upd(const Wt<T>& k, Cx<T> ax, Cx<T> f0, Cx<T> bq, Cx<T>* rhs) {
    if (MODE == P_SWEEP) return fma_c(k.dinv, bq - ax, f0);
    if (MODE == P_RESID) return bq - ax;
    *rhs = fma_c(k.alpha, ax, cmul(k.beta, bq));
    return cmul(k.dinv, *rhs);
}

// Item d of a pass, complex64.  src, dst: iterates; bsrc: the right side (P_HSS: r), bdst: where
// P_HSS writes it; both point one row before the first own row, so that one offset fits all.
// An inner tile: columns x, x + 1 and up to TR rows.
template <int MODE, int TR, bool REP>
__device__ __forceinline__ void tile_pair(const Wt<float>& k, unsigned d, int W, const float2* src, float2* dst,
                                          const float2* bsrc, float2* bdst, const Push& ps) {
    using C = Cx<float>;
    const int at = d & kOff, rows = rows_of(d);
    C h0[TR + 2], h1[TR + 2], a[TR + 2], b[TR + 2];
    if (MODE != P_FIRST) {
#pragma unroll
        for (int t = 0; t < TR + 2; ++t) {
            const float2* p = src + at + (TR <= 2 ? t - 1 : min(t - 1, rows)) * W;
            const float4 o = *reinterpret_cast<const float4*>(p);
            const float2 l = p[-1], r = p[2];
            a[t] = C{o.x, o.y};
            b[t] = C{o.z, o.w};
            h0[t] = C{l.x, l.y} + b[t];
            h1[t] = a[t] + C{r.x, r.y};
        }
    }
#pragma unroll
    for (int t = 1; t <= TR; ++t) {
        if (TR > 1 && t > rows) break;
        const int o = at + (t - 1) * W;
        const float4 bb = *reinterpret_cast<const float4*>(bsrc + o);
        C v0, v1, rhs0, rhs1;
        if (MODE == P_FIRST) {
            v0 = cmul(k.dinv, C{bb.x, bb.y});
            v1 = cmul(k.dinv, C{bb.z, bb.w});
        } else {
            const C e0 = h0[t] + (a[t - 1] + a[t + 1]), e1 = h1[t] + (b[t - 1] + b[t + 1]);
            const C d0 = h0[t - 1] + h0[t + 1], d1 = h1[t - 1] + h1[t + 1];
            const C ax0 = fma_c(k.w[2], d0, fma_c(k.w[1], e0, cmul(k.w[0], a[t])));
            const C ax1 = fma_c(k.w[2], d1, fma_c(k.w[1], e1, cmul(k.w[0], b[t])));
            v0 = upd<float, MODE>(k, ax0, a[t], C{bb.x, bb.y}, &rhs0);
            v1 = upd<float, MODE>(k, ax1, b[t], C{bb.z, bb.w}, &rhs1);
        }
        if (d & kTwo) {
            if (MODE == P_HSS) st_pair(bdst + o, rhs0, rhs1);
            st_pair(dst + o, v0, v1);
        } else {
            if (MODE == P_HSS) st<float>(bdst, o, rhs0);
            st<float>(dst, o, v0);
        }
        if (!REP && (d & (kUp | kDn))) {
            const bool su = (d & kUp) && t == 1, sd = (d & kDn) && t == rows;
            if (d & kTwo) {
                if (su) send2(ps.up + o * 8, v0, v1, ps.bup);
                if (sd) send2(ps.dn + o * 8, v0, v1, ps.bdn);
            } else {
                if (su) send(ps.up + o * 8, v0, ps.bup);
                if (sd) send(ps.dn + o * 8, v0, ps.bdn);
            }
        }
    }
}

// a boundary node
template <int MODE, bool REP>
__device__ __forceinline__ void tile_side(const Wt<float>& k, unsigned d, int W, const float2* src, float2* dst,
                                          const float2* bsrc, float2* bdst, const Push& ps) {
    using C = Cx<float>;
    const int at = d & kOff;
    C v = C{0, 0}, rhs;
    if (!(d & kVoid)) {
        const C bq = ld<float>(bsrc, at);
        if (MODE == P_FIRST) {
            v = cmul(k.dinv, bq);
        } else {
            const float2* p = src + at;
            const C f0 = ld<float>(p, 0);
            const C hx = ld<float>(p, -1) + ld<float>(p, 1), vy = ld<float>(p, -W) + ld<float>(p, W);
            const C dg = (ld<float>(p, -W - 1) + ld<float>(p, -W + 1)) + (ld<float>(p, W - 1) + ld<float>(p, W + 1));
            const C ax = fma_c(k.w[3], dg, fma_c(k.w[2], vy, fma_c(k.w[1], hx, cmul(k.w[0], f0))));
            v = upd<float, MODE>(k, ax, f0, bq, &rhs);
        }
        if (MODE == P_HSS) st<float>(bdst, at, rhs);
        st<float>(dst, at, v);
    }
    if (!REP && (d & (kUp | kDn))) {
        if (d & kUp) send(ps.up + at * 8, v, ps.bup);
        if (d & kDn) send(ps.dn + at * 8, v, ps.bdn);
    }
}

template <int MODE, int TR, bool REP>
__device__ __forceinline__ void tile(const Wt<float>& k, unsigned d, int W, const float2* src, float2* dst,
                                     const float2* bsrc, float2* bdst, const Push& ps) {
    if (!(d & kValid)) return;
    if (kind_of(d) == 8)
        tile_pair<MODE, TR, REP>(k, d, W, src, dst, bsrc, bdst, ps);
    else
        tile_side<MODE, REP>(k, d, W, src, dst, bsrc, bdst, ps);
}

// Item d of a pass, complex128: one node, part `q` (0 real, 1 imaginary) by this lane and the other
// by its neighbour lane.  The whole warp runs it (items without kValid store nothing), and all
// items of a warp are inner or all are on a side.  c * own + i-part: w.re own + wi other with
// wi = -+ w.im gives each part of cmul and fma_c with their own roundings.
__device__ __forceinline__ void send1(unsigned dst, double v, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(dst), "d"(v), "r"(bar)
                 : "memory");
}
struct Half {
    int q;
    __device__ __forceinline__ double wi(Cx<double> c) const { return q ? c.im : -c.im; }
    __device__ __forceinline__ double mul(Cx<double> c, double own, double oth) const {
        return fma(c.re, own, wi(c) * oth);
    }
    __device__ __forceinline__ double mad(Cx<double> c, double own, double oth, double acc) const {
        return fma(c.re, own, fma(wi(c), oth, acc));
    }
};
template <int MODE, int TR, bool REP>
__device__ __forceinline__ void tile(const Wt<double>& k, unsigned d, int W, const double2* src2, double2* dst2,
                                     const double2* bsrc2, double2* bdst2, const Push& ps) {
    const int q = threadIdx.x & 1, at = 2 * (int)(d & kOff) + q, W2 = 2 * W;
    const Half H{q};
    const double* p = reinterpret_cast<const double*>(src2) + at;
    const double* bp = reinterpret_cast<const double*>(bsrc2) + at;
    const int ot = 1 - 2 * q;  // the other part, relative to ours
    const double bq = bp[0];
    auto other = [](double v) { return __shfl_xor_sync(0xffffffffu, v, 1); };
    double v, rhs = 0.0;
    if (MODE == P_FIRST) {
        v = H.mul(k.dinv, bq, bp[ot]);
    } else {
        const double f0 = p[0];
        const double hx = p[-2] + p[2], vy = p[-W2] + p[W2];
        const double dg = (p[-W2 - 2] + p[-W2 + 2]) + (p[W2 - 2] + p[W2 + 2]);
        double ax = H.mul(k.w[0], f0, p[ot]);
        const double dgo = other(dg);
        if (kind_of(d) == 8) {
            const double e = hx + vy;
            ax = H.mad(k.w[1], e, other(e), ax);
            ax = H.mad(k.w[2], dg, dgo, ax);
        } else {
            ax = H.mad(k.w[1], hx, other(hx), ax);
            ax = H.mad(k.w[2], vy, other(vy), ax);
            ax = H.mad(k.w[3], dg, dgo, ax);
        }
        if (MODE == P_HSS) {
            rhs = H.mad(k.alpha, ax, other(ax), H.mul(k.beta, bq, bp[ot]));
            v = H.mul(k.dinv, rhs, other(rhs));
        } else {
            const double r = bq - ax;
            v = MODE == P_SWEEP ? H.mad(k.dinv, r, other(r), f0) : r;
        }
    }
    if (!(d & kValid)) return;
    if (d & kVoid) {
        v = 0.0;
    } else {
        if (MODE == P_HSS) reinterpret_cast<double*>(bdst2)[at] = rhs;
        reinterpret_cast<double*>(dst2)[at] = v;
    }
    if (!REP && (d & (kUp | kDn))) {
        if (d & kUp) send1(ps.up + at * 8, v, ps.bup);
        if (d & kDn) send1(ps.dn + at * 8, v, ps.bdn);
    }
}

template <typename T>
__device__ __forceinline__ const unsigned* words() {
    return reinterpret_cast<const unsigned*>(vecs<T>());
}
// lanes per item: complex128 splits a node over two
template <typename T> constexpr int kLanes = sizeof(T) == 4 ? 1 : 2;

// The items of level L that this thread takes in every pass.  A small level has at most one per
// thread: the item and its weights are then read once for the passes that follow each other.
template <typename T> struct Mine {
    bool one;
    unsigned d;
    Wt<T> k;
};
template <typename T, int MODE>
__device__ __forceinline__ Mine<T> mine(const Lev& L, const PCoef<T>& c) {
    Mine<T> m;
    m.one = L.tiles * kLanes<T> <= kResThreads;
    m.d = m.one && (int)threadIdx.x < L.tiles * kLanes<T> ? words<T>()[L.t0 + threadIdx.x / kLanes<T>] : 0u;
    m.k = weights<T, MODE>(c, kind_of(m.d));
    return m;
}

// one pass (src -> dst: offsets of iterates; bsrc: of the right side)
template <typename T, int MODE, int TR, bool REP>
__device__ __forceinline__ void run(Res& S, const Lev& L, const PCoef<T>& c, const Mine<T>& m, int src, int dst, int bsrc) {
    vec2<T>* const sm = vecs<T>();
    Push ps{};
    if (!REP) {
        ps = push_rows<T>(S, L, dst);
        pass_begin<T>(S, L);
    }
    vec2<T>* const bdst = sm + L.b - L.W;
    if (m.one) {
        // (complex128 items exchange parts between lanes: whole warps, all of a kind)
        if (sizeof(T) == 4 || (int)(threadIdx.x & ~31u) < L.tiles * kLanes<T>)
            tile<MODE, TR, REP>(m.k, m.d, L.W, sm + src, sm + dst, sm + bsrc - L.W, bdst, ps);
    } else {
        const unsigned* dw = words<T>() + L.t0;
        for (int it = threadIdx.x; it < L.tiles * kLanes<T>; it += kResThreads) {
            const unsigned d = dw[it / kLanes<T>];
            const Wt<T> k = weights<T, MODE>(c, kind_of(d));
            tile<MODE, TR, REP>(k, d, L.W, sm + src, sm + dst, sm + bsrc - L.W, bdst, ps);
        }
    }
    if (REP) {
        __syncthreads();
    } else {
        pass_end<T>(S, L);
    }
}

// SECOND < 0: one pass of mode FIRST, src -> dst.  Else two: FIRST src -> dst, SECOND dst -> src.
template <typename T, int FIRST, int SECOND, int TR, bool REP>
__device__ __forceinline__ void run_two(Res& S, const Lev& L, const PCoef<T>& c, int src, int dst, int bsrc) {
    const Mine<T> m = mine<T, FIRST>(L, c);
    run<T, FIRST, TR, REP>(S, L, c, m, src, dst, bsrc);
    if constexpr (SECOND >= 0) {
        if (!REP && S.dead()) return;
        run<T, SECOND, TR, REP>(S, L, c, m, dst, src, bsrc);
    }
}

// The same for level `lvl` with coefficient record `ci`; returns S.round.
template <typename T, int FIRST, int SECOND>
__device__ __noinline__ int passes(Res S, int lvl, int ci, int src, int dst, int bsrc) {
    if (S.dead()) return S.round;
    const Lev L = head<T>().lv[lvl];
    const PCoef<T>& c = head<T>().coef[ci];
    if (L.rep) {
        if (sizeof(T) == 8 || L.tr == 1) run_two<T, FIRST, SECOND, 1, true>(S, L, c, src, dst, bsrc);
        else run_two<T, FIRST, SECOND, 4, true>(S, L, c, src, dst, bsrc);
    } else {
        if (sizeof(T) == 8 || L.tr == 1) run_two<T, FIRST, SECOND, 1, false>(S, L, c, src, dst, bsrc);
        else if (L.tr == 2) run_two<T, FIRST, SECOND, 2, false>(S, L, c, src, dst, bsrc);
        else run_two<T, FIRST, SECOND, 4, false>(S, L, c, src, dst, bsrc);
    }
    return S.round;
}

// Full-weighting restriction of the residual in level lvl's A into b of level lvl + 1, and that
// level's first sweep from 0 into its A.  `copies`: the number of right sides sent to the
// replicated levels so far.
template <typename T>
__device__ __noinline__ int restrict_pass(Res S, int lvl, int copies) {
    Head<T>& hd = head<T>();
    const Lev L = hd.lv[lvl], M = hd.lv[lvl + 1];
    const bool spread = M.rep && !L.rep && S.cs > 1;  // the level's right side goes to every CTA
    // every CTA is done with the last right side, ours (whose rows the loop below overwrites) included
    if (spread) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (S.dead()) return S.round;
    const PCoef<T>& c = hd.coef[lvl + 1];
    vec2<T>* const sm = vecs<T>();
    const Push ps = push_rows<T>(S, M, M.A);
    pass_begin<T>(S, M);
    if (spread && threadIdx.x == 0) {
        hd.copies = copies + 1;
        bar_expect(saddr(&hd.mbr[copies & 1]), (unsigned)((M.nn - M.bulkn) * M.W * sizeof(vec2<T>)));
    }
    const uint2* dw = reinterpret_cast<const uint2*>(words<T>() + M.r0);
    for (int it = threadIdx.x; it < M.restricted; it += kResThreads) {
        // x: offset of fine node (2I, 2J - 1) in A, and of coarse node (I, J) in an iterate << 16
        const uint2 d = dw[it];
        const int at = d.x >> 16, kind = kind_of(d.y);
        Cx<T> x1 = cx<T>(0, 0);
        if (!(d.y & kVoid)) {  // (elsewhere b and both iterates stay 0)
            const vec2<T>* p = sm + L.A + (d.x & kOff);
            const Cx<T> di = kind == 8 ? c.wdinv : c.bdinv[kind];
            Cx<T> acc;
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                const Cx<T> l = ld<T>(p, t * L.W - 1), m = ld<T>(p, t * L.W), r = ld<T>(p, t * L.W + 1);
                const Cx<T> rr = fma_r(T(0.5), l + r, m);
                if (t == 0) acc = half_rn(rr);
                else if (t == 1) acc = acc + rr;
                else acc = fma_r(T(0.5), rr, acc);
            }
            st<T>(sm, M.b - M.W + at, acc);
            if (!spread) {
                x1 = cmul(di, acc);
                st<T>(sm, M.A + at, x1);
            }
        }
        if (d.y & kUp) send(ps.up + at * (unsigned)sizeof(vec2<T>), x1, ps.bup);
        if (d.y & kDn) send(ps.dn + at * (unsigned)sizeof(vec2<T>), x1, ps.bdn);
    }
    if (!spread) {
        if (M.rep) __syncthreads();
        else pass_end<T>(S, M);
        return S.round;
    }
    // our rows of the right side to every other CTA
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if ((int)threadIdx.x < S.cs && (int)threadIdx.x != S.rank && M.bulkn > 0) {
        const unsigned src = saddr(sm + M.b + M.bulk0 * M.W), bytes = (unsigned)(M.bulkn * M.W * sizeof(vec2<T>));
        asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         remote(src, threadIdx.x)),
                     "r"(src), "r"(bytes), "r"(remote(saddr(&hd.mbr[copies & 1]), threadIdx.x))
                     : "memory");
    }
    if (threadIdx.x == 0 && !bounded_wait(&hd.mbr[copies & 1], (copies >> 1) & 1, S.spin)) hd.gave_up[2] = kDead;
    __syncthreads();
    return S.round | hd.gave_up[2];
}

// The coarsest level: its first sweep is in A, the last one has to end in B.
template <typename T, int TR, bool REP>
__device__ __forceinline__ void sweeps(Res& S, const Lev& L, const PCoef<T>& c, int nsweeps, int& src, int& dst) {
    const Mine<T> m = mine<T, P_SWEEP>(L, c);
    for (int s = 1; s < nsweeps; ++s) {
        run<T, P_SWEEP, TR, REP>(S, L, c, m, src, dst, L.b);
        const int t = src;
        src = dst;
        dst = t;
        if (!REP && S.dead()) return;
    }
}
template <typename T>
__device__ __noinline__ int coarse_sweeps(Res S, int lvl, int nsweeps) {
    if (S.dead()) return S.round;
    const Lev L = head<T>().lv[lvl];
    const PCoef<T>& c = head<T>().coef[lvl];
    int src = L.A, dst = L.B;
    if (L.rep) {
        if (sizeof(T) == 8 || L.tr == 1) sweeps<T, 1, true>(S, L, c, nsweeps, src, dst);
        else sweeps<T, 4, true>(S, L, c, nsweeps, src, dst);
    } else {
        if (sizeof(T) == 8 || L.tr == 1) sweeps<T, 1, false>(S, L, c, nsweeps, src, dst);
        else if (L.tr == 2) sweeps<T, 2, false>(S, L, c, nsweeps, src, dst);
        else sweeps<T, 4, false>(S, L, c, nsweeps, src, dst);
    }
    if (src != L.B) {  // an odd number of sweeps
        vec2<T>* const sm = vecs<T>();
        for (int q = threadIdx.x; q < (L.R + 2) * L.W; q += kResThreads) st<T>(sm, L.B + q, ld<T>(sm, L.A + q));
        __syncthreads();
    }
    return S.round;
}

// B of level lvl += P e, e the iterate in B of level lvl + 1, on our rows and the halo rows
template <typename T>
__device__ __noinline__ void prolong_pass(const Res S, int lvl) {
    if (S.dead()) return;
    const Lev& L = head<T>().lv[lvl];
    const Lev& M = head<T>().lv[lvl + 1];
    vec2<T>* const sm = vecs<T>();
    const vec2<T>* const eb = sm + M.B;
    vec2<T>* const xb = sm + L.B;
    const int W = L.W, Wc = M.W, cells = L.cells;
    const uint2* dw = reinterpret_cast<const uint2*>(words<T>() + L.p0);
    for (int it = threadIdx.x; it < cells; it += kResThreads) {
        // x: offset of coarse node (q, J) and, << 16, of fine node (2q + 1, 2J + 1); y: bit t * 2 + h
        // set: fine node (2q + 1 + h, 2J + t) is written.  (Columns and rows beside the level read as 0,
        // or their values, from elsewhere in shared memory, are not used.)
        const uint2 d = dw[it];
        const vec2<T>* e = eb + (d.x & kOff);
        vec2<T>* x = xb + (d.x >> 16);
        const Cx<T> c00 = ld<T>(e, 0), c10 = ld<T>(e, 1), c01 = ld<T>(e, Wc), c11 = ld<T>(e, Wc + 1);
        const Cx<T> x0 = ld<T>(x, -W), x1 = ld<T>(x, 1 - W), x2 = ld<T>(x, 0), x3 = ld<T>(x, 1);
        const Cx<T> m0 = half_rn(c00 + c10), m1 = half_rn(c01 + c11);
        if (d.y & 1) st<T>(x, -W, x0 + m0);
        if (d.y & 2) st<T>(x, 1 - W, x1 + c10);
        if (d.y & 4) st<T>(x, 0, x2 + half_rn(m0 + m1));
        if (d.y & 8) st<T>(x, 1, x3 + half_rn(c10 + c11));
    }
    __syncthreads();
}

// A value of another CTA's shared memory, at the address of our own copy.
__device__ __forceinline__ int peer(const int* p, int rank) {
    int v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(remote(saddr(p), rank)) : "memory");
    return v;
}

// A cluster in which a wait ran out, after the cluster barrier behind its passes (every CTA has sent what it
// will): a CTA that gave up waits for what is still on its way to it, so that none of it arrives after the
// CTA has left.  Of the halo rows that is its last pass's, if the neighbour sent them, and those of one
// pass more, in which the neighbour gave up for want of our rows (hence its row_bytes); of the right
// sides (of level lr) the last one's from the CTAs that sent it, and the next one's.
template <typename T>
__device__ __noinline__ void give_up(const Res S, int lr) {
    Head<T>& hd = head<T>();
    const int copies = hd.copies;
    constexpr unsigned long long kDrain = 4194304;  // (microseconds are enough)
    const int r = S.round & ~kDead;
    if ((threadIdx.x == 0 && S.rank > 0) || (threadIdx.x == 32 && S.rank + 1 < S.cs)) {
        const int d = threadIdx.x == 0 ? 0 : 1, q = S.rank + 2 * d - 1;
        const int sent = peer(&hd.rounds, q);
        if (r > 0 && sent >= r) bounded_wait(&hd.mb[d][(r - 1) & 1], ((r - 1) >> 1) & 1, kDrain);
        if (sent > r) {
            bar_expect(saddr(&hd.mb[d][r & 1]), (unsigned)peer(&hd.row_bytes, q));
            bounded_wait(&hd.mb[d][r & 1], (r >> 1) & 1, kDrain);
        }
    }
    if (threadIdx.x == 64 && lr > 0) {
        unsigned missing = 0, next = 0;
        for (int q = 0; q < S.cs; ++q) {
            if (q == S.rank) continue;
            const unsigned bytes = (unsigned)(peer(&hd.lv[lr].bulkn, q) * hd.lv[lr].W * (int)sizeof(vec2<T>));
            const int sent = peer(&hd.copies, q);
            if (sent < copies) missing += bytes;
            if (sent > copies) next += bytes;
        }
        if (copies > 0) {
            unsigned long long* bar = &hd.mbr[(copies - 1) & 1];
            if (missing)
                asm volatile("mbarrier.complete_tx.relaxed.cluster.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar)),
                             "r"(missing)
                             : "memory");
            bounded_wait(bar, ((copies - 1) >> 1) & 1, kDrain);
        }
        if (next) {
            bar_expect(saddr(&hd.mbr[copies & 1]), next);
            bounded_wait(&hd.mbr[copies & 1], (copies >> 1) & 1, kDrain);
        }
    }
}

// ---- set-up: the levels and their item words ----
// Items of a pass over R rows of a level with n + 1 columns, `rows` of them inner, `edges` the
// level's first or last row: tr rows per inner tile, inner tiles, their end rounded to a warp,
// boundary nodes, all items in whole warps.
struct ResItems {
    int tr, inner, top, side, tiles;
};
template <typename T>
__host__ __device__ inline ResItems resident_items(int n, int R, int rows, int edges) {
    const int unit = sizeof(T) == 4 ? 32 : 16, cols = sizeof(T) == 4 ? n >> 1 : n - 1;
    ResItems t;
    t.side = 2 * R + edges * (n - 1);
    t.tr = 1;
    if (sizeof(T) == 4) {
        // the fewest rows per thread that still finish in one round (parallelism first), else 4
        // (fewest shared-memory reads per node)
        const int room = kResThreads - ((t.side + 31) & ~31);
        if (rows * cols > room) t.tr = ((rows + 1) / 2) * cols <= room ? 2 : 4;
    }
    t.inner = ((rows + t.tr - 1) / t.tr) * cols;
    t.top = (t.inner + unit - 1) / unit * unit;
    t.tiles = t.top + (t.side + unit - 1) / unit * unit;
    return t;
}

// class of node (i, j): 8 inner, else its boundary class
__device__ __forceinline__ unsigned node_kind(int n, int i, int j) {
    const int tx = i == 0 ? 0 : (i == n ? 2 : 1), ty = j == 0 ? 0 : (j == n ? 2 : 1);
    return tx == 1 && ty == 1 ? 8u : (unsigned)bclass2(tx, ty);
}
__device__ __forceinline__ unsigned send_flags(const Lev& L, int rl) {
    return (L.up && rl == 0 ? kUp : 0u) | (L.dn && rl == L.R - 1 ? kDn : 0u);
}

// Level l of the CTA with rows f0 .. f1 - 1 (fu: the CTA above starts there).
template <typename T>
__device__ Lev make_level(const ResArgs<T>& a, int l, int f0, int f1, int fu) {
    const int nn = a.lv[l].nn, n = nn - 1;
    Lev L;
    L.rep = l >= a.dist;
    L.nn = nn;
    L.W = a.lv[l].W;
    L.row0 = L.rep ? 0 : f0;
    L.R = L.rep ? nn : f1 - f0;
    L.Ru = f0 - fu;
    L.A = a.lv[l].offA;
    L.B = a.lv[l].offB;
    L.b = a.lv[l].offb;
    L.up = !L.rep && L.row0 > 0;
    L.dn = !L.rep && L.row0 + L.R < nn;
    L.bulk0 = f0;
    L.bulkn = f1 - f0;
    L.t0 = a.lv[l].offt;
    L.r0 = a.lv[l].offr;
    L.p0 = a.lv[l].offp;
    const int lo = L.row0 == 0 ? 1 : 0, hi = L.row0 + L.R == nn ? L.R - 2 : L.R - 1;
    const ResItems t = resident_items<T>(n, L.R, max(hi - lo + 1, 0), (lo ? 1 : 0) + (hi == L.R - 2 ? 1 : 0));
    L.tr = t.tr;
    L.tiles = t.tiles;
    // (a replicated level that the distributed one above restricts to: only our rows)
    L.restricted = (L.rep && (l > a.dist || a.dist == 0) ? nn : f1 - f0) * nn;
    if (l == 0) L.restricted = 0;
    const int jlo = max(L.row0 - (L.rep ? 0 : 1), 0), jhi = min(L.row0 + L.R - (L.rep ? 1 : 0), n);
    L.cells = l + 1 < a.levels ? ((jhi >> 1) - (jlo >> 1) + 1) * ((n >> 1) + 1) : 0;
    return L;
}

template <typename T>
__device__ void make_words(const ResArgs<T>& a, const Res& S, int l) {
    unsigned* const wd = reinterpret_cast<unsigned*>(vecs<T>());
    const Lev L = head<T>().lv[l];
    const int n = L.nn - 1, W = L.W;
    auto voidn = [&](int m, int i, int j) {
        return (i == 0 && (S.dir & 1)) || (i == m && (S.dir & 2)) || (j == 0 && (S.dir & 4)) || (j == m && (S.dir & 8));
    };
    // tiles: the inner nodes by groups of tr rows, then the boundary nodes (columns 0 and n of each
    // row, then rows 0 and n where owned), each part padded to whole warps
    const int lo = L.row0 == 0 ? 1 : 0, hi = L.row0 + L.R == L.nn ? L.R - 2 : L.R - 1, rows = max(hi - lo + 1, 0);
    const int cols = sizeof(T) == 4 ? n >> 1 : n - 1;
    const ResItems t = resident_items<T>(n, L.R, rows, (lo ? 1 : 0) + (hi == L.R - 2 ? 1 : 0));
    for (int it = threadIdx.x; it < t.tiles; it += kResThreads) {
        unsigned d;
        if (it < t.top) {
            const bool ok = it < t.inner;
            const int g = ok ? it / cols : 0, q = ok ? it - g * cols : 0, rl = lo + g * t.tr;
            const int nr = ok ? min(t.tr, hi - rl + 1) : 1, i = sizeof(T) == 4 ? 2 * q + 1 : q + 1;
            d = (unsigned)((ok ? rl + 1 : 1) * W + i + 1) | (unsigned)nr << 16 | 8u << 22;
            if (ok)
                d |= kValid | (i + 1 < n ? kTwo : 0u) | (send_flags(L, rl) & kUp) | (send_flags(L, rl + nr - 1) & kDn);
        } else {
            int q = it - t.top, i = 0, rl = 0;
            const bool ok = q < t.side;
            if (ok) {
                if (q < 2 * L.R) {
                    i = (q & 1) ? n : 0;
                    rl = q >> 1;
                } else {
                    q -= 2 * L.R;
                    const bool first = lo && q < n - 1;
                    i = (lo && !first ? q - (n - 1) : q) + 1;
                    rl = first ? 0 : L.R - 1;
                }
            }
            d = (unsigned)((rl + 1) * W + i + 1) | 1u << 16 | (ok ? node_kind(n, i, L.row0 + rl) : 0u) << 22;
            if (ok) d |= kValid | send_flags(L, rl) | (voidn(n, i, L.row0 + rl) ? kVoid : 0u);
        }
        wd[L.t0 + it] = d;
    }
    if (l > 0) {
        // nodes restricted from the finer level: rows J whose centre row the CTA owns there
        const Lev F = head<T>().lv[l - 1];
        const int J0 = (F.row0 + 1) >> 1;
        for (int it = threadIdx.x; it < L.restricted; it += kResThreads) {
            const int Jl = it / L.nn, I = it - Jl * L.nn, J = J0 + Jl, rl = J - L.row0;
            const unsigned fine = (unsigned)((2 * J - F.row0) * F.W + 2 * I + 1);
            const unsigned y = (unsigned)node_kind(n, I, J) << 22 | (voidn(n, I, J) ? kVoid : 0u) | send_flags(L, rl);
            reinterpret_cast<uint2*>(wd + L.r0)[it] = make_uint2(fine | (unsigned)((rl + 1) * W + I + 1) << 16, y);
        }
    }
    if (l + 1 < a.levels) {
        const Lev M = head<T>().lv[l + 1];
        const int jlo = max(L.row0 - (L.rep ? 0 : 1), 0), jhi = min(L.row0 + L.R - (L.rep ? 1 : 0), n);
        const int pc = (n >> 1) + 1;
        for (int it = threadIdx.x; it < L.cells; it += kResThreads) {
            const int cj = it / pc, q = it - cj * pc - 1, J = (jlo >> 1) + cj;
            unsigned y = 0;
            for (int h = 0; h < 4; ++h) {
                const int i = 2 * q + 1 + (h & 1), j = 2 * J + (h >> 1);
                if (i >= 0 && i <= n && j >= jlo && j <= jhi && !voidn(n, i, j)) y |= 1u << h;
            }
            const unsigned e = (unsigned)((J - M.row0 + 1) * M.W + q + 1);
            reinterpret_cast<uint2*>(wd + L.p0)[it] =
                make_uint2(e | (unsigned)((2 * J - L.row0 + 2) * W + 2 * q + 2) << 16, y);
        }
    }
}

}  // namespace

// grid: cs CTAs per problem, problem blockIdx.x / cs.  HSS: z = the HSS loop's result for r
// (complex128 in and out); else x = one cycle on A_L x = b from 0 (vectors in T).
template <typename T, bool HSS>
__global__ void __launch_bounds__(kResThreads, 1) k_resident2(const __grid_constant__ ResArgs<T> a) {
    // (the kernels behind this one may not come before its end: parked on the free SMs for the length of an HSS
    // loop, their blocks kept the clusters of other streams, which want 16 SMs to themselves, from starting.
    // 48 uneven solves per second on four worker slots / in one pack: 15.9 / 34.4 so, 33.6 / 57.5 now)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int prob = blockIdx.x / a.cs;
    if (a.active && !a.active[prob]) return;  // uniform over the cluster
    Head<T>& hd = head<T>();
    vec2<T>* const sm = vecs<T>();
    Res S;
    S.cs = a.cs;
    S.rank = (int)blockIdx.x - prob * a.cs;  // (clusters are runs of cs consecutive CTAs)
    S.dir = (a.dir[0] ? 1 : 0) | (a.dir[1] ? 2 : 0) | (a.dir[2] ? 4 : 0) | (a.dir[3] ? 8 : 0);
    S.round = 0;
    S.spin = a.spin_limit;
    // what goes up arrives as the upper neighbour's row from below, and the other way round
    const int ru = S.rank > 0 ? S.rank - 1 : 0, rd = S.rank + 1 < S.cs ? S.rank + 1 : S.rank;
    S.base_up = remote(saddr(sm), ru);
    S.base_dn = remote(saddr(sm), rd);
    S.mb_up = remote(saddr(&hd.mb[1][0]), ru);
    S.mb_dn = remote(saddr(&hd.mb[0][0]), rd);
    const int Lc = a.levels;
    for (int q = threadIdx.x; q < a.elems; q += kResThreads) st<T>(sm, q, cx<T>(0, 0));
    for (int l = 0; l <= Lc; ++l) {
        const PCoef<T>* src = l < Lc ? a.al + (long long)l * a.nb + prob : a.ar + prob;
        const unsigned* w = reinterpret_cast<const unsigned*>(src);
        unsigned* d = reinterpret_cast<unsigned*>(&hd.coef[l]);
        if (l < Lc || HSS)
            for (int q = threadIdx.x; q < (int)(sizeof(PCoef<T>) / 4); q += kResThreads) d[q] = w[q];
    }
    if (threadIdx.x == 0) {
        for (int q = 0; q < 4; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&hd.mb[q >> 1][q & 1])) : "memory");
        for (int q = 0; q < 2; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&hd.mbr[q])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        hd.gave_up[0] = hd.gave_up[1] = hd.gave_up[2] = hd.any = hd.copies = 0;
    } else if (threadIdx.x == 32) {
        const int nn0 = a.lv[0].nn;
        int f0 = S.rank * nn0 / a.cs, f1 = (S.rank + 1) * nn0 / a.cs, fu = S.rank > 0 ? (S.rank - 1) * nn0 / a.cs : 0;
        for (int l = 0; l < Lc; ++l) {
            hd.lv[l] = make_level<T>(a, l, f0, f1, fu);
            f0 = (f0 + 1) >> 1;
            f1 = (f1 + 1) >> 1;
            fu = (fu + 1) >> 1;
        }
    }
    __syncthreads();
    for (int l = 0; l < Lc; ++l) make_words<T>(a, S, l);
    const Lev L0 = hd.lv[0];
    const int nn0 = L0.nn;
    // r of the HSS steps (kept in shared memory, or where that is full converted to r_lo and read
    // into the free iterate A at every step), or the cycle's right side
    const bool keep = !HSS || a.off_r >= 0;
    const int rin = !HSS ? L0.b : keep ? a.off_r : L0.A + L0.W;
    const long long base = (long long)prob * nn0 * nn0 + (long long)L0.row0 * nn0;
    for (int q = threadIdx.x; q < L0.R * nn0; q += kResThreads) {
        const int rl = q / nn0, i = q - rl * nn0;
        Cx<T> v;
        if constexpr (HSS) {
            const double2 d = a.r[base + q];
            // (0 at Dirichlet nodes, which the iterate A, where r may be read to, has to hold)
            const int j = L0.row0 + rl, n0 = nn0 - 1;
            const bool vd = (i == 0 && a.dir[0]) || (i == n0 && a.dir[1]) || (j == 0 && a.dir[2]) || (j == n0 && a.dir[3]);
            v = vd ? cx<T>(0, 0) : cx<T>(T(d.x), T(d.y));
        } else {
            v = ld<T>(a.b, base + q);
        }
        if (keep)
            st<T>(sm, rin + rl * L0.W + i + 1, v);
        else
            st<T>(a.r_lo, base + q, v);
    }
    // every CTA's buffers and barriers are set before any halo row or copy arrives
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (a.cs > 1) cg::this_cluster().sync(); else __syncthreads();
    const bool copies = a.cs > 1 && a.dist < Lc;  // replicated levels fed by the cluster
    if (copies) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");

    const int steps = HSS ? a.nhss[prob] : 1;
    for (int it = 0; it < steps; ++it) {
        if (HSS) {
            if (!keep) {
                for (int q = threadIdx.x; q < L0.R * nn0; q += kResThreads) {
                    const int rl = q / nn0, i = q - rl * nn0;
                    st<T>(sm, rin + rl * L0.W + i + 1, ld<T>(a.r_lo, base + q));
                }
                __syncthreads();
            }
            S.round = passes<T, P_HSS, -1>(S, 0, Lc, L0.B, L0.A, rin);
        } else {
            S.round = passes<T, P_FIRST, -1>(S, 0, 0, L0.A, L0.A, L0.b);
        }
        for (int l = 0; l < Lc - 1; ++l) {
            S.round = passes<T, P_SWEEP, P_RESID>(S, l, l, hd.lv[l].A, hd.lv[l].B, hd.lv[l].b);
            S.round = restrict_pass<T>(S, l, it);
            if (copies && l + 1 == a.dist)
                passes<T, P_FIRST, -1>(S, l + 1, l + 1, hd.lv[l + 1].A, hd.lv[l + 1].A, hd.lv[l + 1].b);
        }
        S.round = coarse_sweeps<T>(S, Lc - 1, a.nu_coarse);
        for (int l = Lc - 2; l >= 0; --l) {
            prolong_pass<T>(S, l);
            // (the replicated levels' right side is not read any more)
            if (copies && l == a.dist - 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
            S.round = passes<T, P_SWEEP, P_SWEEP>(S, l, l, hd.lv[l].B, hd.lv[l].A, hd.lv[l].b);
        }
    }
    if (copies) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    auto write = [&](long long p, Cx<T> v) {
        if constexpr (HSS)
            a.z[p] = make_double2((double)v.re, (double)v.im);
        else
            st<T>(a.x, p, v);
    };
    for (int q = threadIdx.x; q < L0.R * nn0; q += kResThreads) {
        const int rl = q / nn0, i = q - rl * nn0;
        write(base + q, ld<T>(sm, L0.B + (rl + 1) * L0.W + i + 1));
    }
    if (a.cs == 1) return;
    if (threadIdx.x == 0) {
        hd.rounds = S.round & ~kDead;
        if (S.dead()) *a.status = HSS ? kLoopTimeout : kCycleTimeout;
    }
    if (S.dead() && (int)threadIdx.x < S.cs)
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote(saddr(&hd.any), threadIdx.x)), "r"(1) : "memory");
    cg::this_cluster().sync();  // nobody leaves while another may still send to it
    if (hd.any) {
        if (S.dead()) give_up<T>(S, copies ? a.dist : 0);
        // no half-finished result: a single cycle's caller is told only by its next blocking call
        for (int q = threadIdx.x; q < L0.R * nn0; q += kResThreads) write(base + q, cx<T>(T(NAN), T(NAN)));
        __syncthreads();
        cg::this_cluster().sync();
    }
}

namespace {

// Rows of each level for clusters of cs CTAs, distributed levels and shared-memory layout;
// false when the level set does not fit.
template <typename T>
bool plan_for(ResArgs<T>* P, const GridDesc* lv, int levels, bool hss, int cs) {
    // a level of at most so many nodes costs less computed by every CTA than distributed
    const long long rep_nodes = sizeof(T) == 4 ? 1100 : 100;
    P->cs = cs;
    P->levels = levels;
    P->dist = 0;
    std::vector<int> f(cs + 1);
    for (int r = 0; r <= cs; ++r) f[r] = (int)((long long)r * lv[0].nn / cs);
    size_t e = 0;
    int tiles[kResMaxLevels] = {0}, restricted[kResMaxLevels] = {0}, cells[kResMaxLevels] = {0};
    size_t bs0 = 0;
    for (int l = 0; l < levels; ++l) {
        const int nn = lv[l].nn, n = nn - 1;
        if (l < levels - 1 && (n & 1)) return false;
        const bool dist = cs > 1 && lv[l].N > rep_nodes && P->dist == l;
        if (dist) P->dist = l + 1;
        int rows = 0;
        for (int r = 0; r < cs; ++r) {
            const int own = f[r + 1] - f[r];
            if (dist && own < 1) return false;
            const int r0 = dist ? f[r] : 0, R = dist ? own : nn;
            const bool first = r0 == 0, last = r0 + R == nn;
            const ResItems t = resident_items<T>(n, R, std::max(R - first - last, 0), first + last);
            const int jlo = std::max(r0 - (dist ? 1 : 0), 0), jhi = std::min(r0 + R - (dist ? 0 : 1), n);
            rows = std::max(rows, R);
            tiles[l] = std::max(tiles[l], t.tiles);
            restricted[l] = std::max(restricted[l], (dist || l == P->dist ? own : nn) * nn);
            cells[l] = std::max(cells[l], ((jhi >> 1) - (jlo >> 1) + 1) * ((n >> 1) + 1));
        }
        const int W = (nn + 2) & ~1;  // even: rows and pairs of columns start on 16 bytes
        const size_t it = (size_t)(rows + 2) * W + 2, bs = (size_t)rows * W + 2;
        if (it + W > 0xffff) return false;  // (item words hold 16-bit offsets)
        P->lv[l].nn = nn;
        P->lv[l].W = W;
        P->lv[l].offA = (int)e;
        P->lv[l].offB = (int)(e + it);
        P->lv[l].offb = (int)(e + 2 * it);
        e += 2 * it + bs;
        if (l == 0) bs0 = bs;
        for (int r = 0; r <= cs; ++r) f[r] = (f[r] + 1) >> 1;
    }
    if (cs > 1 && P->dist == 0) return false;  // nothing to distribute: one CTA is enough
    size_t w = 0;  // words
    for (int l = 0; l < levels; ++l) {
        P->lv[l].offt = (int)w;
        w += (tiles[l] + 1) & ~1;
        P->lv[l].offr = (int)w;
        if (l > 0) w += 2 * (size_t)restricted[l];
        P->lv[l].offp = (int)w;
        if (l + 1 < levels) w += 2 * (size_t)cells[l];
    }
    P->off_r = -1;
    if (hss && kHead<T> + (e + bs0) * sizeof(vec2<T>) + w * 4 <= kResSmemMax) {
        P->off_r = (int)e;
        e += bs0;
    }
    const size_t base = e * sizeof(vec2<T>) / 4;
    for (int l = 0; l < levels; ++l) {
        P->lv[l].offt += (int)base;
        P->lv[l].offr += (int)base;
        P->lv[l].offp += (int)base;
    }
    P->elems = (int)e;
    P->smem = kHead<T> + e * sizeof(vec2<T>) + w * 4;
    return P->smem <= kResSmemMax;
}

// Configure k_resident2<T, HSS>; active[q]: clusters of 16, 8, 4, 2 CTAs that the device holds at
// once with the largest shared memory.
template <typename T, bool HSS>
cudaError_t prepare_one(int (&active)[4]) {
    cudaError_t e = cudaFuncSetAttribute(k_resident2<T, HSS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kResSmemMax);
    if (e != cudaSuccess) return e;
    cudaFuncSetAttribute(k_resident2<T, HSS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaGetLastError();
    for (int q = 0; q < 4; ++q) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(16u >> q);
        cfg.blockDim = dim3(kResThreads);
        cfg.dynamicSmemBytes = kResSmemMax;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 16u >> q;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        active[q] = 0;
        if (cudaOccupancyMaxActiveClusters(&active[q], k_resident2<T, HSS>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            active[q] = 0;
        }
    }
    return cudaSuccess;
}

}  // namespace

template <typename T>
bool resident_plan(ResArgs<T>* P, const GridDesc* lv, int levels, int nb, bool hss) {
    if (levels < 2 || levels > kResMaxLevels || lv[0].dim != 2) return false;
    // per device: clusters of 16, 8, 4, 2 CTAs held at once (set-up under a lock, once)
    constexpr int kMaxDev = 64;
    static std::mutex mu;
    static int state[kMaxDev], held[kMaxDev][4];
    int dev = 0, active[4];
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
        cudaGetLastError();
        return false;
    }
    {
        std::lock_guard<std::mutex> g(mu);
        if (state[dev] == 0) {
            int a1[4], a0[4];
            state[dev] = -1;
            if (prepare_one<T, true>(a1) == cudaSuccess && prepare_one<T, false>(a0) == cudaSuccess) {
                state[dev] = 1;
                for (int q = 0; q < 4; ++q) held[dev][q] = std::min(a1[q], a0[q]);
            }
            cudaGetLastError();
        }
        if (state[dev] < 0) return false;
        for (int q = 0; q < 4; ++q) active[q] = held[dev][q];
    }
    P->nb = nb;
    for (int q = 0; q < 4; ++q) P->dir[q] = lv[0].dir[q];
    // the largest clusters (a problem's cycle is shortest with them) that the device holds at once: a batch in
    // several waves of clusters would be slower than the separate kernels over all its problems.  HSS step of a
    // batch, us, here / separate: complex64 65^2 8 problems (16 CTAs) 15.7 / 45, 32 (4) 16.9 / 51, 64 (2)
    // 19.7 / 60, 152 (1) 20.6 / 89; 97^2 76 (2) 28 / 84; 129^2 9 (8) 22 / 47, 36 (4) 28 / 77; 257^2 7 (16) 30 / 56;
    // complex128 33^2 128 (1) 98 / 425, 65^2 64 (2) 180 / 459, 97^2 32 (4) 206 / 417, 129^2 8 (8) 186 / 279
    for (int q = 0; q < 4; ++q)
        if (active[q] >= nb && plan_for<T>(P, lv, levels, hss, 16 >> q)) return true;
    return nb <= num_sms() && plan_for<T>(P, lv, levels, hss, 1);
}

template <typename T>
cudaError_t launch_resident(const ResArgs<T>& P, bool hss, cudaStream_t s) {
    const dim3 grd((unsigned)(P.cs * P.nb)), blk(kResThreads);
    if (hss) return klaunch(k_resident2<T, true>, grd, blk, P.smem, s, P.cs, P);
    return klaunch(k_resident2<T, false>, grd, blk, P.smem, s, P.cs, P);
}

template bool resident_plan<float>(ResArgs<float>*, const GridDesc*, int, int, bool);
template bool resident_plan<double>(ResArgs<double>*, const GridDesc*, int, int, bool);
template cudaError_t launch_resident<float>(const ResArgs<float>&, bool, cudaStream_t);
template cudaError_t launch_resident<double>(const ResArgs<double>&, bool, cudaStream_t);

}  // namespace hh
