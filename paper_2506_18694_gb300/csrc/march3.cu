// 3D fused V-cycle kernels.  A CTA of 8 warps owns a tile of 30 x-nodes, 8 consecutive
// y-rows (the first and last are halo rows) and R + 2 consecutive z-planes (the first and
// last are halo planes); it writes the 30 x 6 x R interior outputs.  Warp w loads its row
// of every plane with one coalesced access per plane (all loads in flight before any
// arithmetic), forms the x-neighbour sum by warp shuffles, and publishes the value and the
// x-sum of each plane in shared memory; after one barrier the six output warps read rows
// j-1 and j+1 from shared memory and keep their own row in registers.  Interior nodes use
// the four neighbour-class weights of the 27-point Q1 operator (centre, face, edge,
// corner).  The field is loaded as zero outside the cube and at Dirichlet nodes, so a node
// on a face, edge or corner sums its existing neighbours by group (centre; x, y, z faces;
// xy, xz, yz edges; corners) with the eight weights of its boundary class.
//
// Bound by the shared-memory pipe (257^3 Jacobi sweep: its wavefronts 76 % busy, issue 52 %), then by the
// loads' latency at 32 warps per SM.  On that sweep and on that grid's V-cycle, us: complex sums as packed
// adds and no boundary checks in the output warps 118 -> 113; tiles off every face (72 %) compiled without
// any check 113 -> 109, 769 -> 740; value and x-sum side by side, one 16-byte access for both, 109 -> 107,
// 703 -> 685 (129^3 HSS step 162 -> 154).
#include "internal.h"

namespace hh {

namespace {

template <typename T>
__device__ __forceinline__ Cx<T> shfl_up3(Cx<T> v) {
    return Cx<T>{__shfl_up_sync(0xffffffffu, v.re, 1), __shfl_up_sync(0xffffffffu, v.im, 1)};
}
template <typename T>
__device__ __forceinline__ Cx<T> shfl_dn3(Cx<T> v) {
    return Cx<T>{__shfl_down_sync(0xffffffffu, v.re, 1), __shfl_down_sync(0xffffffffu, v.im, 1)};
}

// Whether coordinate v of an axis with Dirichlet flags lo, hi holds no unknown.
__device__ __forceinline__ bool void1(int v, int n, int lo, int hi) {
    return v < 0 || v > n || (v == 0 && lo) || (v == n && hi);
}

__device__ __forceinline__ int type1(int v, int n) { return v <= 0 ? 0 : (v >= n ? 2 : 1); }

// Boundary-class index of a node with axis types tx, ty, tz (not all inner).
__device__ __forceinline__ int bclass3(int tx, int ty, int tz) {
    const int c = (tz * 3 + ty) * 3 + tx;
    return c - (c > 13);
}

// Window of a node: the field value (f*) and x-neighbour sum (x*) of its column on planes
// l-1, l, l+1, and the sums over rows j-1 and j+1 of the value (vy*) and of the x-sum (sy*).
template <typename T> struct Win3 {
    Cx<T> fm, f0, fp, xm, x0, xp, vy0, vy1, vy2, sy0, sy1, sy2;
};

// The output of one node (offset p) from its window: the 27-point product A x assembled by
// neighbour group, then the mode's update.  FAST: an interior node (the four weights of the
// interior stencil); else the eight group weights of the node's boundary class (tx, ty, l).
template <typename T, int MODE, bool FAST>
__device__ __forceinline__ void out3(const MArgs<T>& a, const PCoef<T>& cf, const Cx<T>* bw, const VPtrs<T>& v,
                                     const Win3<T>& q, Cx<T> zq, int tx, int ty, int l, bool cvoid, long long p) {
    const int n = a.g.n;
    Cx<T> ax, dinv_w;
    bool masked = false;
    if (FAST) {
        const Cx<T> face = q.x0 + q.vy1 + (q.fm + q.fp);
        const Cx<T> edge = q.sy1 + (q.xm + q.xp) + (q.vy0 + q.vy2);
        const Cx<T> corner = q.sy0 + q.sy2;
        ax = fma_c(cf.iw[3], corner, fma_c(cf.iw[2], edge, fma_c(cf.iw[1], face, cmul(cf.iw[0], q.f0))));
        dinv_w = cf.wdinv;
    } else {
        // neighbour groups: centre; x, y, z faces; xy, xz, yz edges; corners
        masked = cvoid || void1(l, n, a.g.dir[4], a.g.dir[5]);
        const Cx<T>* wq = bw + bclass3(tx, ty, type1(l, n)) * kClass3Len;
        ax = cmul(wq[0], q.f0);
        ax = fma_c(wq[1], q.x0, ax);
        ax = fma_c(wq[2], q.vy1, ax);
        ax = fma_c(wq[3], q.fm + q.fp, ax);
        ax = fma_c(wq[4], q.sy1, ax);
        ax = fma_c(wq[5], q.xm + q.xp, ax);
        ax = fma_c(wq[6], q.vy0 + q.vy2, ax);
        ax = fma_c(wq[7], q.sy0 + q.sy2, ax);
        dinv_w = wq[8];
    }
    const Cx<T> alpha = a.use_pc_ab ? cf.alpha : a.alpha, beta = a.use_pc_ab ? cf.beta : a.beta;
    if (masked) {
        st<T>(v.y, p, cx<T>(0, 0));
        if (MODE == M_HSS_FIRST) st<T>(v.y2, p, cx<T>(0, 0));
    } else if (MODE == M_APPLY) {
        st<T>(v.y, p, ax);
    } else if (MODE == M_AXPBY) {
        st<T>(v.y, p, fma_c(alpha, ax, cmul(beta, zq)));
    } else if (MODE == M_DAXPBY) {
        st<T>(v.y, p, cmul(dinv_w, fma_c(alpha, ax, cmul(beta, zq))));
    } else if (MODE == M_HSS_FIRST) {
        const Cx<T> rhs = fma_c(alpha, ax, cmul(beta, zq));
        st<T>(v.y, p, rhs);
        st<T>(v.y2, p, cmul(dinv_w, rhs));
    } else {
        st<T>(v.y, p, fma_c(dinv_w, zq - ax, q.f0));
    }
}

// Field value and x-neighbour sum of a node, side by side: one shared-memory access for both (of 16 bytes
// in complex64).
template <typename T> struct __align__(16) Pair3 {
    vec2<T> v, s;
};

constexpr int kWarps3 = 8;  // y-rows per tile, including the two halo rows

}  // namespace

// One tile.  Nodes outside the cube and Dirichlet nodes load as zero: one predicate per column and a
// uniform one per plane.  Output rows and planes are uniform over a warp, so a warp runs either the
// inner formula or that of one boundary class; the columns i = 0 and n, where lanes would differ, are
// left to the two halo warps, which have nothing to do after the barrier: a lane per node, from the
// sums in shared memory.  INNER: every node the tile loads lies inside the cube, off every face, and
// no check is made at all.
template <typename T, int MODE, int R, bool BATCH, bool INNER>
__device__ __forceinline__ void march3_tile(const MArgs<T>& a, int b, int bx, int by, int l0,
                                            unsigned char* smem_raw) {
    const PCoef<T>& cf = BATCH ? a.pc[b] : a.c0;
    const Cx<T>* bw = a.bw3 + (long long)b * kClass3 * kClass3Len;
    const VPtrs<T> v = problem_ptrs(a, b, false);
    constexpr int NP = R + 2;  // planes loaded
    constexpr bool NEEDZ = MODE != M_APPLY;
    Pair3<T>* const sm = reinterpret_cast<Pair3<T>*>(smem_raw);  // [warp][plane][lane]
    const int lane = threadIdx.x & 31;
    const int w = threadIdx.x >> 5;
    const int n = a.g.n, nn = a.g.nn;
    const int i = bx * 30 + lane - 1;
    const int j = by * (kWarps3 - 2) + w - 1;
    const bool cvoid = !INNER && (void1(i, n, a.g.dir[0], a.g.dir[1]) || void1(j, n, a.g.dir[2], a.g.dir[3]));
    const bool zero = cvoid || (MODE != M_JACOBI2_ZERO && a.xzero);
    const int tx = INNER ? 1 : type1(i, n), ty = INNER ? 1 : type1(j, n);
    const long long ps = (long long)nn * nn;
    const long long col = (long long)j * nn + i + l0 * ps;  // (used where the node lies in the cube)
    const vec2<T>* const xin = (MODE == M_JACOBI2_ZERO ? v.z : v.x) + col;

    Cx<T> fv[NP], xs[NP];
#pragma unroll
    for (int t = 0; t < NP; ++t) {
        const int l = l0 - 1 + t;
        fv[t] = (zero || (!INNER && void1(l, n, a.g.dir[4], a.g.dir[5]))) ? cx<T>(0, 0) : ld<T>(xin, (t - 1) * ps);
    }
    const bool out_row = w >= 1 && w <= kWarps3 - 2;
    const bool out = out_row && lane >= 1 && lane <= 30 && (INNER || (tx == 1 && j <= n));
    Cx<T> zv[R];
#pragma unroll
    for (int t = 0; t < R; ++t)
        zv[t] = (NEEDZ && out && (INNER || l0 + t <= n)) ? ld<T>(v.z + col, t * ps) : cx<T>(0, 0);
    if (MODE == M_JACOBI2_ZERO) {
        // first sweep from x = 0: x1 = omega D^{-1} b
        const bool in = tx == 1 && ty == 1;
#pragma unroll
        for (int t = 0; t < NP; ++t) {
            const int l = l0 - 1 + t;
            const Cx<T> d = INNER || (in && l >= 1 && l <= n - 1) ? cf.wdinv : bw[bclass3(tx, ty, type1(l, n)) * kClass3Len + 8];
            fv[t] = cmul(d, fv[t]);
        }
    }
#pragma unroll
    for (int t = 0; t < NP; ++t) {
        xs[t] = shfl_up3(fv[t]) + shfl_dn3(fv[t]);
        Pair3<T> e;
        e.v.x = fv[t].re;
        e.v.y = fv[t].im;
        e.s.x = xs[t].re;
        e.s.y = xs[t].im;
        sm[(w * NP + t) * 32 + lane] = e;
    }
    __syncthreads();
    if (INNER && !out_row) return;
    if (!out_row) {
        // column i = 0 (warp 0) or n (the last warp), if the tile holds it: rows by * 6 + r, planes l0 + t
        const int is = w == 0 ? 0 : n, lc = is - bx * 30 + 1;
        if (lc < 1 || lc > 30) return;
        for (int q = lane; q < (kWarps3 - 2) * R; q += 32) {
            const int r = q / R, t = q - r * R, js = by * (kWarps3 - 2) + r, l = l0 + t;
            if (js > n || l > n) continue;
            const int e = ((r + 1) * NP + t) * 32 + lc;  // its row on plane l - 1
            constexpr int P = 32, Y = NP * 32;
            const long long p = (long long)js * nn + is + l * ps;
            const Cx<T> zq = NEEDZ ? ld<T>(v.z, p) : cx<T>(0, 0);
            auto fv1 = [&](int o) { const vec2<T> u = sm[e + o].v; return cx<T>(u.x, u.y); };
            auto xs1 = [&](int o) { const vec2<T> u = sm[e + o].s; return cx<T>(u.x, u.y); };
            const Win3<T> q3{fv1(0), fv1(P), fv1(2 * P), xs1(0), xs1(P), xs1(2 * P),
                             fv1(-Y) + fv1(Y), fv1(P - Y) + fv1(P + Y), fv1(2 * P - Y) + fv1(2 * P + Y),
                             xs1(-Y) + xs1(Y), xs1(P - Y) + xs1(P + Y), xs1(2 * P - Y) + xs1(2 * P + Y)};
            const bool vd = void1(is, n, a.g.dir[0], a.g.dir[1]) || void1(js, n, a.g.dir[2], a.g.dir[3]);
            out3<T, MODE, false>(a, cf, bw, v, q3, zq, type1(is, n), type1(js, n), l, vd, p);
        }
        return;
    }
    if (!out) return;
    const int wm = w - 1, wp = w + 1;
    // rows j-1 + j+1 summed (value and x-sum) per plane, in a rolling window of 3 planes
    auto ysum = [&](int tpl, Cx<T>& vy, Cx<T>& sy) {
        const Pair3<T> m = sm[(wm * NP + tpl) * 32 + lane], p = sm[(wp * NP + tpl) * 32 + lane];
        vy = cx<T>(m.v.x, m.v.y) + cx<T>(p.v.x, p.v.y);
        sy = cx<T>(m.s.x, m.s.y) + cx<T>(p.s.x, p.s.y);
    };
    Win3<T> q;
    ysum(0, q.vy0, q.sy0);
    ysum(1, q.vy1, q.sy1);
    const long long p0 = col;
#pragma unroll
    for (int t = 0; t < R; ++t) {
        const int l = l0 + t;
        if (!INNER && l > n) break;
        const int tp = t + 1;  // local plane of the output
        ysum(tp + 1, q.vy2, q.sy2);
        q.fm = fv[tp - 1];
        q.f0 = fv[tp];
        q.fp = fv[tp + 1];
        q.xm = xs[tp - 1];
        q.x0 = xs[tp];
        q.xp = xs[tp + 1];
        const long long p = p0 + t * ps;
        if (INNER || (ty == 1 && l >= 1 && l <= n - 1))  // (uniform over the warp)
            out3<T, MODE, true>(a, cf, bw, v, q, zv[t], 1, 1, l, false, p);
        else
            out3<T, MODE, false>(a, cf, bw, v, q, zv[t], 1, ty, l, cvoid, p);
        q.vy0 = q.vy1;
        q.vy1 = q.vy2;
        q.sy0 = q.sy1;
        q.sy1 = q.sy2;
    }
}

// BATCH = false: a batch of one, coefficients from the kernel parameters, no activity flags.
template <typename T, int MODE, int R, bool BATCH>
__global__ void __launch_bounds__(32 * kWarps3, sizeof(T) == 4 && R <= 4 ? 4 : 1) k_march3(const __grid_constant__ MArgs<T> a, int zt) {
    pdl_entry();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = BATCH ? (int)blockIdx.z / zt : 0;  // problem; blockIdx.z % zt: z-tile
    if (BATCH && problem_skipped(a, b)) return;
    const int l0 = (blockIdx.z - b * zt) * R, n = a.g.n;
    const int i0 = (int)blockIdx.x * 30 - 1, j0 = (int)blockIdx.y * (kWarps3 - 2) - 1, z0 = l0 - 1;
    if (i0 >= 1 && i0 + 31 <= n - 1 && j0 >= 1 && j0 + kWarps3 - 1 <= n - 1 && z0 >= 1 && z0 + R + 1 <= n - 1)
        march3_tile<T, MODE, R, BATCH, true>(a, b, blockIdx.x, blockIdx.y, l0, smem_raw);
    else
        march3_tile<T, MODE, R, BATCH, false>(a, b, blockIdx.x, blockIdx.y, l0, smem_raw);
}

// Weights of the 3D boundary classes.  1D rows (Q1): stiffness (1/h)(-1, cnt, -1), mass
// (h/6)(1, 2 cnt, 1), cnt = 2 inside and 1 at the ends of the axis.  Group S (the axes along
// which the neighbour is offset) has stiffness weight sum_a K_a prod_{b != a} M_b and mass
// weight prod_b M_b, with K_a, M_b the side weights (-1/h, h/6) on offset axes and the
// centre weights otherwise; a node on the side of axis a also carries the 2D boundary mass
// of that face, prod_{b != a} M_b, for the groups not offset along a.
template <typename T>
void boundary_weights3(Cx<T>* out, const PCoef<T>& c, const GridDesc& g, double omega) {
    const double h = g.h, ks = -1.0 / h, ms = h / 6.0;
    // groups: centre; x, y, z faces; xy, xz, yz edges; corners (bit a set: offset along axis a)
    const int groups[8] = {0, 1, 2, 4, 3, 5, 6, 7};
    for (int tz = 0; tz < 3; ++tz)
        for (int ty = 0; ty < 3; ++ty)
            for (int tx = 0; tx < 3; ++tx) {
                const int cl = (tz * 3 + ty) * 3 + tx;
                if (cl == 13) continue;
                const int q = cl - (cl > 13);
                const int typ[3] = {tx, ty, tz};
                double kc[3], mc[3];
                for (int a = 0; a < 3; ++a) {
                    const double cnt = typ[a] == 1 ? 2.0 : 1.0;
                    kc[a] = cnt / h;
                    mc[a] = cnt * h / 3.0;
                }
                double A[8], M[8], F[8];
                for (int u = 0; u < 8; ++u) {
                    const int S = groups[u];
                    double kk[3], mm[3];
                    for (int a = 0; a < 3; ++a) {
                        const bool off = (S >> a) & 1;
                        kk[a] = off ? ks : kc[a];
                        mm[a] = off ? ms : mc[a];
                    }
                    A[u] = kk[0] * mm[1] * mm[2] + mm[0] * kk[1] * mm[2] + mm[0] * mm[1] * kk[2];
                    M[u] = mm[0] * mm[1] * mm[2];
                    F[u] = 0.0;
                    for (int a = 0; a < 3; ++a)
                        if (typ[a] != 1 && !((S >> a) & 1)) F[u] += mm[(a + 1) % 3] * mm[(a + 2) % 3];
                }
                Cx<T>* o = out + (size_t)q * kClass3Len;
                for (int u = 0; u < 8; ++u)
                    o[u] = cx<T>(T(double(c.op.cK) * A[u] + double(c.op.cM.re) * M[u] + double(c.op.cG.re) * F[u]),
                                 T(double(c.op.cM.im) * M[u] + double(c.op.cG.im) * F[u]));
                const double dr = double(c.opd.cK) * A[0] + double(c.opd.cM.re) * M[0] + double(c.opd.cG.re) * F[0];
                const double di = double(c.opd.cM.im) * M[0] + double(c.opd.cG.im) * F[0];
                const double d2 = dr * dr + di * di;
                o[8] = d2 > 0 ? cx<T>(T(omega * dr / d2), T(-omega * di / d2)) : cx<T>(T(0), T(0));
            }
}

template void boundary_weights3<float>(Cx<float>*, const PCoef<float>&, const GridDesc&, double);
template void boundary_weights3<double>(Cx<double>*, const PCoef<double>&, const GridDesc&, double);

template <typename T, int MODE, int R>
static cudaError_t go3(MArgs<T> a, cudaStream_t s) {
    // at most 40 KiB: within the default dynamic shared-memory limit, no opt-in needed
    const size_t smem = 2 * (size_t)kWarps3 * (R + 2) * 32 * sizeof(vec2<T>);
    static_assert(2 * kWarps3 * (R + 2) * 32 * sizeof(vec2<T>) <= 48 * 1024, "tile too large");
    const int zt = (a.g.nn + R - 1) / R;
    const int tx = (a.g.nn + 29) / 30, ty = (a.g.nn + kWarps3 - 3) / (kWarps3 - 2);
    dim3 grd((unsigned)tx, (unsigned)ty, (unsigned)(zt * a.nb));
    if (a.pc) return klaunch(k_march3<T, MODE, R, true>, grd, dim3(32 * kWarps3), smem, s, 1, a, zt);
    if (a.nb != 1) return cudaErrorInvalidValue;
    return klaunch(k_march3<T, MODE, R, false>, grd, dim3(32 * kWarps3), smem, s, 1, a, zt);
}

// Planes per tile of the complex64 kernels (the results do not depend on them).  4 where the grid fills
// the chip (257^3: 8 halve the resident CTAs, 2 double the halo planes); a grid of few tiles is bound by
// the chain of one tile, which shortens with its planes.  HSS step of the 3D preconditioner with 4, 2, 1
// planes on every level, us: 41^3 72, 58, 53; 49^3 74, 61, 62 (234 tiles of 4); 65^3 79, 74, 77 (561);
// 97^3 108, 110 (1700); 129^3 168, 200.
int march3_planes(const GridDesc& g, int nb) {
    const long long nn = g.nn, sms = num_sms();
    const long long tiles = ((nn + 29) / 30) * ((nn + kWarps3 - 3) / (kWarps3 - 2)) * ((nn + 3) / 4) * nb;
    return 3 * tiles <= 4 * sms ? 1 : (tiles <= 2 * sms ? 2 : 4);
}

template <typename T, int MODE>
static cudaError_t pick3(MArgs<T> a, cudaStream_t s) {
    a.h = T(a.g.h);
    a.ih = T(1.0 / a.g.h);
    if constexpr (sizeof(T) == 4) {
        switch (a.tile_rows ? a.tile_rows : march3_planes(a.g, a.nb)) {
            case 1: return go3<T, MODE, 1>(a, s);
            case 2: return go3<T, MODE, 2>(a, s);
            case 8: return go3<T, MODE, 8>(a, s);
            default: return go3<T, MODE, 4>(a, s);
        }
    } else {
        return go3<T, MODE, 2>(a, s);
    }
}

template <typename T>
cudaError_t launch_march3(int mode, const MArgs<T>& a, cudaStream_t s) {
    if (a.g.dim != 3) return cudaErrorInvalidValue;
    switch (mode) {
        case M_APPLY: return pick3<T, M_APPLY>(a, s);
        case M_AXPBY: return pick3<T, M_AXPBY>(a, s);
        case M_DAXPBY: return pick3<T, M_DAXPBY>(a, s);
        case M_JACOBI: return pick3<T, M_JACOBI>(a, s);
        case M_HSS_FIRST: return pick3<T, M_HSS_FIRST>(a, s);
        case M_JACOBI2_ZERO: return pick3<T, M_JACOBI2_ZERO>(a, s);
        default: return cudaErrorInvalidValue;
    }
}

template cudaError_t launch_march3<float>(int, const MArgs<float>&, cudaStream_t);
template cudaError_t launch_march3<double>(int, const MArgs<double>&, cudaStream_t);

}  // namespace hh
