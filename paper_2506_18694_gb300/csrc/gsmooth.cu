// Vector kernels of the GMRES smoother (Sec. 5.3: GMRES with a Jacobi preconditioner on
// every level).  One smoothing step of s iterations on A x = b from x runs, with
// M = omega D^{-1} A applied by the stencil kernels' M_DAXPBY mode:
//   z0 = omega D^{-1} (b - A x), beta = ||z0||, v_0 = z0 / beta;
//   for j < s: w = M v_j; two passes of classical Gram-Schmidt against v_0..v_j (the
//   coefficients of both passes added into column j of H); h_{j+1,j} = ||w||, v_{j+1} = w / h,
//   and column j reduced by Givens rotations (as in GMRES, one new rotation per step);
//   y = R^{-1} g minimises ||beta e1 - H y||; x += V y.
// Inner products and norms are summed in the level precision within a block (FP64 arithmetic
// is slow on this part and the complex64 smoother does not need it) and the block shares are
// combined in FP64: each block writes its share, and the kernel that uses a sum adds the
// shares in a fixed order (every block of that kernel the same way), so the result is the
// same whatever ran before and however the problems are batched.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <mutex>

#include "internal.h"
#include "march2_common.cuh"

namespace cg = cooperative_groups;

namespace hh {

namespace {

__device__ __forceinline__ bool gs_skip(const Batch& bt, int b) {
    if (bt.active && !bt.active[b]) return true;
    return bt.hss_it >= 0 && bt.hss_it >= bt.nhss[b];
}

__device__ __forceinline__ double2 dadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

// fused multiply-add in the level precision (FP64 arithmetic, conversions included, runs on
// this part's narrow FP64 pipe: kept out of the per-element loops of the complex64 smoother)
__device__ __forceinline__ float fmaT(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmaT(double a, double b, double c) { return fma(a, b, c); }

// sum of every thread's acc[i] (i < nv) over the block into out[i] (as FP64), by warp
// butterflies and then the warps in order; sh holds kGsThreads / 32 * kGsMaxVec entries
template <typename T>
__device__ void block_sums(Cx<T> (&acc)[kGsMaxVec], int nv, Cx<T>* sh, double2* out) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < kGsMaxVec; ++i) {
        if (i >= nv) break;
        Cx<T> v = acc[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            v.re += __shfl_xor_sync(0xffffffffu, v.re, o);
            v.im += __shfl_xor_sync(0xffffffffu, v.im, o);
        }
        if (lane == 0) sh[wid * kGsMaxVec + i] = v;
    }
    __syncthreads();
    if ((int)threadIdx.x < nv) {
        Cx<T> t = cx<T>(0, 0);
        for (int w = 0; w < kGsThreads / 32; ++w) t = t + sh[w * kGsMaxVec + threadIdx.x];
        out[threadIdx.x] = make_double2(t.re, t.im);
    }
}

// sum of n block shares p[0], p[stride], ... by one warp: lane t adds shares t, t + 32, ...
// in order, then the lanes are combined by a fixed butterfly (the same order on every call)
__device__ __forceinline__ double2 warp_sum_shares(const double2* p, int n, int stride) {
    const int lane = threadIdx.x & 31;
    double2 t = make_double2(0.0, 0.0);
    for (int k = lane; k < n; k += 32) t = dadd(t, p[(long long)k * stride]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        t.x += __shfl_xor_sync(0xffffffffu, t.x, o);
        t.y += __shfl_xor_sync(0xffffffffu, t.y, o);
    }
    return t;
}

// grid (nblk, nb)
template <typename T>
__global__ void __launch_bounds__(kGsThreads) k_gs_dot(const vec2<T>* __restrict__ V, long long ldv, int nv,
                                                       const vec2<T>* __restrict__ w, long long N,
                                                       double2* __restrict__ part, Batch bt) {
    pdl_entry();
    const int b = blockIdx.y;
    if (gs_skip(bt, b)) return;
    __shared__ Cx<T> sh[kGsThreads / 32 * kGsMaxVec];
    const vec2<T>* Vb = V + (long long)b * N;
    const vec2<T>* wb = w + (long long)b * N;
    Cx<T> acc[kGsMaxVec];
#pragma unroll
    for (int i = 0; i < kGsMaxVec; ++i) acc[i] = cx<T>(0, 0);
    const long long stride = (long long)gridDim.x * kGsThreads;
    for (long long p = (long long)blockIdx.x * kGsThreads + threadIdx.x; p < N; p += stride) {
        const Cx<T> x = ld<T>(wb, p);
#pragma unroll
        for (int i = 0; i < kGsMaxVec; ++i) {
            if (i >= nv) break;
            const Cx<T> v = ld<T>(Vb + i * ldv, p);
            // conj(v) * x
            acc[i].re = fmaT(v.re, x.re, fmaT(v.im, x.im, acc[i].re));
            acc[i].im = fmaT(v.re, x.im, fmaT(-v.im, x.re, acc[i].im));
        }
    }
    block_sums(acc, nv, sh, part + ((long long)b * gridDim.x + blockIdx.x) * kGsMaxVec);
}

// grid (nblk, nb)
template <typename T>
__global__ void __launch_bounds__(kGsThreads) k_gs_orth(vec2<T>* __restrict__ w, const vec2<T>* __restrict__ V,
                                                        long long ldv, int nv, long long N,
                                                        const double2* __restrict__ part, double2* ls, int col,
                                                        int accumulate, double2* __restrict__ part2, Batch bt) {
    pdl_entry();
    const int b = blockIdx.y;
    if (gs_skip(bt, b)) return;
    __shared__ Cx<T> cneg[kGsMaxVec];  // -c_i in the level precision
    __shared__ Cx<T> sh[kGsThreads / 32 * kGsMaxVec];
    const int nblk = gridDim.x;
    // coefficient i summed by warp i % 8
    for (int i = threadIdx.x >> 5; i < nv; i += kGsThreads / 32) {
        const double2 t = warp_sum_shares(part + (long long)b * nblk * kGsMaxVec + i, nblk, kGsMaxVec);
        if ((threadIdx.x & 31) == 0) {
            cneg[i] = cx<T>(T(-t.x), T(-t.y));
            if (blockIdx.x == 0) {
                double2& h = ls[(long long)b * kGsState + i * kGsMaxIts + col];
                h = accumulate ? dadd(h, t) : t;
            }
        }
    }
    __syncthreads();
    Cx<T> cc[kGsMaxVec];
#pragma unroll
    for (int i = 0; i < kGsMaxVec; ++i) cc[i] = i < nv ? cneg[i] : cx<T>(0, 0);
    vec2<T>* wb = w + (long long)b * N;
    const vec2<T>* Vb = V + (long long)b * N;
    Cx<T> acc[kGsMaxVec];
    acc[0] = cx<T>(0, 0);
    const long long stride = (long long)nblk * kGsThreads;
    for (long long p = (long long)blockIdx.x * kGsThreads + threadIdx.x; p < N; p += stride) {
        Cx<T> x = ld<T>(wb, p);
#pragma unroll
        for (int i = 0; i < kGsMaxVec; ++i) {
            if (i >= nv) break;
            x = fma_c(cc[i], ld<T>(Vb + i * ldv, p), x);
        }
        st<T>(wb, p, x);
        acc[0].re = fmaT(x.re, x.re, fmaT(x.im, x.im, acc[0].re));
    }
    if (part2) block_sums(acc, 1, sh, part2 + ((long long)b * nblk + blockIdx.x) * kGsMaxVec);
}

// complex helpers in the level precision for the small least-squares problem
template <typename T>
__device__ __forceinline__ Cx<T> cget(const double2& d) {
    return cx<T>(T(d.x), T(d.y));
}
template <typename T>
__device__ __forceinline__ double2 cput(Cx<T> v) {
    return make_double2(v.re, v.im);
}
// (p, q) <- (c p + s q, -conj(s) p + c q), c real
template <typename T>
__device__ __forceinline__ void rotate(T c, Cx<T> s, Cx<T>& p, Cx<T>& q) {
    const Cx<T> p0 = p, q0 = q;
    p = cx<T>(c * p0.re + (s.re * q0.re - s.im * q0.im), c * p0.im + (s.re * q0.im + s.im * q0.re));
    q = cx<T>(-(s.re * p0.re + s.im * p0.im) + c * q0.re, -(s.re * p0.im - s.im * p0.re) + c * q0.im);
}

// grid (nblk, nb)
template <typename T>
__global__ void __launch_bounds__(kGsThreads) k_gs_scale(vec2<T>* __restrict__ out, const vec2<T>* __restrict__ w,
                                                         long long N, const double2* __restrict__ part2, int nsum,
                                                         double2* ls, int col, Batch bt) {
    pdl_entry();
    const int b = blockIdx.y;
    if (gs_skip(bt, b)) return;
    __shared__ T inv;
    if (threadIdx.x < 32) {
        const T h = sqrt(T(warp_sum_shares(part2 + (long long)b * nsum * kGsMaxVec, nsum, kGsMaxVec).x));
        if (threadIdx.x == 0) {
            inv = h > T(0) ? T(1) / h : T(0);
            if (blockIdx.x == 0) {
                double2* S = ls + (long long)b * kGsState;
                if (col < 0) {
                    S[kGsRhs] = make_double2(h, 0.0);
                    for (int i = 1; i < kGsMaxVec; ++i) S[kGsRhs + i] = make_double2(0.0, 0.0);
                } else {
                    // column col: previous rotations, then the one that zeroes h = H[col + 1][col]
                    for (int i = 0; i < col; ++i) {
                        Cx<T> p = cget<T>(S[i * kGsMaxIts + col]), q = cget<T>(S[(i + 1) * kGsMaxIts + col]);
                        rotate<T>(T(S[kGsCos + i].x), cget<T>(S[kGsSin + i]), p, q);
                        S[i * kGsMaxIts + col] = cput(p);
                        S[(i + 1) * kGsMaxIts + col] = cput(q);
                    }
                    const Cx<T> a = cget<T>(S[col * kGsMaxIts + col]);
                    const T na = sqrt(a.re * a.re + a.im * a.im);
                    const T den = sqrt(na * na + h * h);
                    T cs = T(1);
                    Cx<T> sn = cx<T>(0, 0);
                    if (den > T(0)) {
                        if (na == T(0)) {
                            cs = T(0);
                            sn = cx<T>(1, 0);
                        } else {
                            // s = (a / |a|) conj(h) / den, h real
                            cs = na / den;
                            sn = cx<T>(a.re / na * h / den, a.im / na * h / den);
                        }
                    }
                    Cx<T> p = a, q = cx<T>(h, 0);
                    rotate<T>(cs, sn, p, q);
                    S[col * kGsMaxIts + col] = cput(p);
                    S[(col + 1) * kGsMaxIts + col] = make_double2(0.0, 0.0);
                    S[kGsCos + col] = make_double2(cs, 0.0);
                    S[kGsSin + col] = cput(sn);
                    Cx<T> g0 = cget<T>(S[kGsRhs + col]), g1 = cget<T>(S[kGsRhs + col + 1]);
                    rotate<T>(cs, sn, g0, g1);
                    S[kGsRhs + col] = cput(g0);
                    S[kGsRhs + col + 1] = cput(g1);
                }
            }
        }
    }
    __syncthreads();
    const T s = inv;
    const vec2<T>* wb = w + (long long)b * N;
    vec2<T>* ob = out + (long long)b * N;
    const long long stride = (long long)gridDim.x * kGsThreads;
    for (long long p = (long long)blockIdx.x * kGsThreads + threadIdx.x; p < N; p += stride) {
        const Cx<T> x = ld<T>(wb, p);
        st<T>(ob, p, cx<T>(x.re * s, x.im * s));
    }
}

// grid (nblk, nb)
template <typename T>
__global__ void __launch_bounds__(kGsThreads) k_gs_update(vec2<T>* __restrict__ x, const vec2<T>* __restrict__ V,
                                                          long long ldv, int m, long long N, const double2* ls,
                                                          int overwrite, Batch bt) {
    pdl_entry();
    const int b = blockIdx.y;
    if (gs_skip(bt, b)) return;
    __shared__ Cx<T> ys[kGsMaxIts];
    if (threadIdx.x == 0) {
        // back substitution R y = g; a zero pivot (breakdown: the space was already
        // invariant) gives y_j = 0
        const double2* S = ls + (long long)b * kGsState;
        for (int j = m - 1; j >= 0; --j) {
            Cx<T> t = cget<T>(S[kGsRhs + j]);
            for (int k = j + 1; k < m; ++k) {
                const Cx<T> r = cget<T>(S[j * kGsMaxIts + k]), yk = ys[k];
                t = cx<T>(t.re - (r.re * yk.re - r.im * yk.im), t.im - (r.re * yk.im + r.im * yk.re));
            }
            const Cx<T> d = cget<T>(S[j * kGsMaxIts + j]);
            const T dd = d.re * d.re + d.im * d.im;
            ys[j] = dd > T(0) ? cx<T>((t.re * d.re + t.im * d.im) / dd, (t.im * d.re - t.re * d.im) / dd)
                              : cx<T>(0, 0);
        }
    }
    __syncthreads();
    Cx<T> yc[kGsMaxIts];
#pragma unroll
    for (int i = 0; i < kGsMaxIts; ++i) yc[i] = i < m ? ys[i] : cx<T>(0, 0);
    vec2<T>* xb = x + (long long)b * N;
    const vec2<T>* Vb = V + (long long)b * N;
    const long long stride = (long long)gridDim.x * kGsThreads;
    for (long long p = (long long)blockIdx.x * kGsThreads + threadIdx.x; p < N; p += stride) {
        Cx<T> acc = overwrite ? cx<T>(0, 0) : ld<T>(xb, p);
#pragma unroll
        for (int i = 0; i < kGsMaxIts; ++i) {
            if (i >= m) break;
            acc = fma_c(yc[i], ld<T>(Vb + i * ldv, p), acc);
        }
        st<T>(xb, p, acc);
    }
}

// ---- the whole smoothing step in one launch: a cluster per problem ----
// Why.  A step of 5 iterations as separate kernels is 34 launches of 3 to 4 us, and in one CTA with the
// basis in global memory it took 85 us on 65^2.  Here (GB300, complex64, 5 iterations) a step takes
// 12 us on 9^2, 18 on 33^2, 24 on 65^2, 33 on 129^2 and 62 on 257^2; the W-cycle of 257^2 went from 2372 to
// 709 us, of 129^2 from 1535 to 528, complex128 129^2 from 9428 to 3419; 16 problems of 129^2 1694 to 845, 64 of
// 2045 to 1810, 64 of 257^2 6164 to 4500, complex128 32 of 129^2 11238 to 9785.  A small level is bound by the
// chain of two sums an iteration (500 cycles in a block, 1350 more for the cluster barrier),
// 257^2 by the shared-memory reads of the basis (four times an iteration).
//
// The Krylov basis of a level lives in the (distributed) shared memory of the cluster, a band of
// rows per CTA with a halo row above and below and a zero column beside the row; w stays in
// registers.  What is left of an iteration is two sums over the cluster, each one cluster barrier.
// The halo rows of w travel with the first; the receiver makes the next basis vector's halo rows
// of them as the sender does its own rows.  The norm comes from the second pass' sums: with c the
// coefficients of that pass and w before it, h^2 = ||w||^2 - ||c||^2, exact to rounding while ||c||^2 is
// a small part of ||w||^2; else (w almost in the space already) it is summed by itself.
//
// Sums: a thread's and a warp's in the level precision; over the warps and the CTAs, in a fixed order, as
// pairs of a sum and its rounding error in complex64 (error-free addition, Knuth's TwoSum).  A coefficient of
// H and the norm are formed from the pairs and rounded once, as the separate kernels form them in FP64,
// which this part does 64 times slower.
template <typename T> struct GsCfg;  // threads a CTA at most
template <> struct GsCfg<float> {
    static constexpr int kThreads = 1024;
};
template <> struct GsCfg<double> {
    static constexpr int kThreads = 512;
};
constexpr int kGsScal = 2 * kGsMaxIts + 1;  // scalars of a sum
// A level takes the fewest CTAs that leave one no more nodes than this (halo rows included), if 16 are
// enough.  W-cycle of 257^2 with GMRES(5), us, for 300, 512, 1024, 2048, 4096 nodes: 756, 751, 785, 793, 932;
// 32 problems of 129^2 together 1281, 1210, 1196, 959, 911; complex128 129^2 3184, 3441, 3827, 4542, 5674.
constexpr int kGsBand = 512;
constexpr int kGsClusterMax = 16;  // (non-portable; fewer where the device does not hold one)
constexpr size_t kGsSmemMax = 226 * 1024;

template <typename T> struct Sum;
template <> struct Sum<float> {
    float hi, lo;
    __device__ static Sum of(float v) { return Sum{v, 0.0f}; }
    // (an infinite or NaN sum makes its rounding error NaN: the sum alone counts then)
    __device__ float value() const { return lo == lo ? hi + lo : hi; }
    __device__ float rest(float v) const {  // what v = value() leaves out
        const float r = __fadd_rn(__fsub_rn(hi, v), lo);
        return r == r ? r : 0.0f;
    }
    __device__ Sum plus_lane(int o) const {
        const float h2 = __shfl_xor_sync(0xffffffffu, hi, o), l2 = __shfl_xor_sync(0xffffffffu, lo, o);
        const float t = __fadd_rn(hi, h2), bb = __fsub_rn(t, hi);
        const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bb)), __fsub_rn(h2, bb));
        return Sum{t, __fadd_rn(__fadd_rn(lo, l2), err)};
    }
};
template <> struct Sum<double> {
    double hi;
    __device__ static Sum of(double v) { return Sum{v}; }
    __device__ double value() const { return hi; }
    __device__ double rest(double) const { return 0.0; }
    __device__ Sum plus_lane(int o) const { return Sum{hi + __shfl_xor_sync(0xffffffffu, hi, o)}; }
};

// (a + la) + (b + lb) rounded once, la and lb small beside a and b
__device__ __forceinline__ float add_pairs(float a, float la, float b, float lb) {
    const float t = __fadd_rn(a, b), bb = __fsub_rn(t, a);
    const float err = __fadd_rn(__fsub_rn(a, __fsub_rn(t, bb)), __fsub_rn(b, bb));
    const float r = __fadd_rn(t, __fadd_rn(err, __fadd_rn(la, lb)));
    return r == r ? r : t;
}
__device__ __forceinline__ double add_pairs(double a, double, double b, double) { return a + b; }

// Weights of a node's kind (boundary class 0..7, 8 inner): centre, x, y and diagonal neighbours,
// omega D^{-1}.
template <typename T> struct alignas(4 * sizeof(T)) GsWeights {
    Cx<T> w[4], dinv, pad;
};

// Start of the dynamic shared memory; the basis vectors follow at kGsHead<T> bytes.
template <typename T> struct GsShared {
    GsWeights<T> wt[9];
    T red[32][kGsScal + 2];  // sums of the warps (a group of sums may end beyond the last vector's)
    Sum<T> part[2][kGsClusterMax][kGsScal];
    // column j at j & 1: its sums (both passes' coefficients; ||w||^2), and what rounding left out of them
    T H[2][2][kGsScal], L[2][2][kGsScal];
    T beta2, tmp, low, h[kGsMaxIts];
    Cx<T> R[kGsMaxIts][kGsMaxIts];
    Cx<T> g[kGsMaxVec], sn[kGsMaxIts], ys[kGsMaxIts];
    T cs[kGsMaxIts];
};
template <typename T> constexpr size_t kGsHead = (sizeof(GsShared<T>) + 127) / 128 * 128;

// A node word: offset in a basis vector, kind, flags (up, dn: sent to that neighbour; free: holds an
// unknown; in: own row, else a halo row).  0: no node; offset 0 is an entry that stays 0.
constexpr unsigned kGsUp = 1u << 20, kGsDn = 1u << 21, kGsFree = 1u << 22, kGsIn = 1u << 23, kGsHalo = 1u << 24;
constexpr unsigned kGsInner = 1u << 25;  // every lane of the warp has an inner node there

template <typename T> struct GsCtx {
    GsShared<T>* sh;
    vec2<T>*vup, *vdn;  // the neighbours' V, shifted so that a sent row's offset is that of their halo row
    vec2<T>* V;         // basis vector i at V + i * ss, row r of the band at (r + 1) * W, column i at + i + 1
    int W, ss, R, rank, cs, phase;
};

// v[0..S) summed over the warp: 32 / S lanes end with each sum; to red[0..S)
template <typename T, int S>
__device__ __forceinline__ void warp_sums(T* v, T* red) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int h = S / 2; h >= 1; h >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const T keep = up ? v[i + h] : v[i], give = up ? v[i] : v[i + h];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
#pragma unroll
    for (; o >= 1; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    if ((lane & (32 / S - 1)) == 0) red[lane / (32 / S)] = v[0];
}

// Column `col` of H, from both passes' sums (added by the lanes of a warp) and the norm h below its
// diagonal: the previous rotations, then the one that zeroes h; the right side g with it (by its lane 0).
template <typename T>
__device__ __forceinline__ void rotate_column(GsShared<T>& s, int col) {
    const int lane = threadIdx.x & 31;
    T(*Hc)[kGsScal] = s.H[col & 1];
    const T(*Lc)[kGsScal] = s.L[col & 1];
    if (lane < 2 * (col + 1)) Hc[0][lane] = add_pairs(Hc[0][lane], Lc[0][lane], Hc[1][lane], Lc[1][lane]);
    __syncwarp();
    if (lane) return;
    auto H = [&](int i) { return cx<T>(Hc[0][2 * i], Hc[0][2 * i + 1]); };
    Cx<T> a = H(0);
    for (int i = 0; i < col; ++i) {
        Cx<T> q = H(i + 1);
        rotate<T>(s.cs[i], s.sn[i], a, q);
        s.R[i][col] = a;
        a = q;
    }
    const T h = s.h[col];
    const T a2 = a.re * a.re + a.im * a.im, na = sqrt(a2), den = sqrt(a2 + h * h);
    T c = T(1);
    Cx<T> sn = cx<T>(0, 0);
    if (den > T(0)) {
        if (na == T(0)) {
            c = T(0);
            sn = cx<T>(1, 0);
        } else {
            // s = (a / |a|) h / den (H's entries are of the order of 1: nothing overflows)
            const T q = h / (na * den);
            c = na / den;
            sn = cx<T>(a.re * q, a.im * q);
        }
    }
    s.cs[col] = c;
    s.sn[col] = sn;
    s.R[col][col] = cx<T>(c * a.re + sn.re * h, c * a.im + sn.im * h);
    const Cx<T> g0 = s.g[col];
    s.g[col] = cx<T>(c * g0.re, c * g0.im);
    s.g[col + 1] = cx<T>(-(sn.re * g0.re + sn.im * g0.im), -(sn.re * g0.im - sn.im * g0.re));
}

// Back substitution R y = g by one warp, row i by lane i; a zero pivot (breakdown: the space was
// already invariant) gives y_j = 0.
template <typename T>
__device__ __forceinline__ void back_substitute(GsShared<T>& s, int its) {
    const int i = threadIdx.x & 31, r = min(i, its - 1);
    Cx<T> t = s.g[r];
    const Cx<T> p = s.R[r][r];
    const T dd = p.re * p.re + p.im * p.im;
    const Cx<T> inv = dd > T(0) ? cx<T>(p.re / dd, -p.im / dd) : cx<T>(0, 0);
    for (int j = its - 1; j >= 0; --j) {
        Cx<T> y = cmul(t, inv);
        y = cx<T>(__shfl_sync(0xffffffffu, y.re, j), __shfl_sync(0xffffffffu, y.im, j));
        if (i == j) s.ys[j] = y;
        if (i < j) t = t - cmul(s.R[i][j], y);
    }
}

// The warps' sums red[.][0..ns) over the cluster into out, and what rounding left out of them into low, the
// same in every CTA.  rot >= 0: while the cluster meets, the last warp reduces column rot by rotations
// (before its arrival the W-cycle of 257^2 took 727 us instead of 709).
template <typename T>
__device__ __forceinline__ void cluster_sums(GsCtx<T>& x, int ns, T* out, T* low, int rot = -1) {
    const int nw = blockDim.x >> 5, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    GsShared<T>& sh = *x.sh;
    __syncthreads();
    Sum<T>(*part)[kGsScal] = sh.part[x.phase & 1];
    for (int q = wid; q < ns; q += nw) {
        Sum<T> t = Sum<T>::of(lane < nw ? sh.red[lane][q] : T(0));
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) t = t.plus_lane(o);  // (every lane ends with the sum)
        if (x.cs == 1) {
            if (lane == 0) low[q] = t.rest(out[q] = t.value());
        } else if (lane < x.cs) {
            *cg::this_cluster().map_shared_rank(&part[x.rank][q], lane) = t;
        }
    }
    const bool rotates = rot >= 0 && threadIdx.x >= blockDim.x - 32;
    if (x.cs == 1) {
        if (rotates) rotate_column<T>(sh, rot);
    } else {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        if (rotates) rotate_column<T>(sh, rot);
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        for (int q = wid; q < ns; q += nw) {
            Sum<T> t = lane < x.cs ? part[lane][q] : Sum<T>::of(T(0));
            for (int o = x.cs >> 1; o >= 1; o >>= 1) t = t.plus_lane(o);
            if (lane == 0) low[q] = t.rest(out[q] = t.value());
        }
        ++x.phase;
    }
    __syncthreads();
}

// op f at a node of a zero-padded band, and omega D^{-1} of the node
template <typename T>
__device__ __forceinline__ Cx<T> band_apply(const GsWeights<T>* wt, const vec2<T>* f, int W, unsigned d, Cx<T>* dinv) {
    const vec2<T>* p = f + (d & 0xffff);
    const GsWeights<T>& k = wt[d & kGsInner ? 8 : (d >> 16) & 15];
    const Cx<T> hx = ld<T>(p, -1) + ld<T>(p, 1), vy = ld<T>(p, -W) + ld<T>(p, W);
    const Cx<T> dg = (ld<T>(p, -W - 1) + ld<T>(p, -W + 1)) + (ld<T>(p, W - 1) + ld<T>(p, W + 1));
    *dinv = k.dinv;
    if (d & kGsInner) {  // (fewer shared loads: 257^2 spends its time on them)
        const GsWeights<T>& c = wt[8];
        return fma_c(c.w[3], dg, fma_c(c.w[1], hx + vy, cmul(c.w[0], ld<T>(p, 0))));
    }
    // (an inner node's four edge neighbours are added first here too, as the stencil kernels do: each product is
    // rounded at the size of the centre's, and a fourth one made the W-cycle's error 3.5 % larger up to 129^2)
    const bool in = ((d >> 16) & 15) == 8;
    const Cx<T> e = in ? hx + vy : hx, v = in ? cx<T>(0, 0) : vy;
    return fma_c(k.w[3], dg, fma_c(k.w[2], v, fma_c(k.w[1], e, cmul(k.w[0], ld<T>(p, 0)))));
}

// w to the neighbours' halo rows of basis vector `to`, and (after a sum) from there
template <typename T, int KN>
__device__ __forceinline__ void send_rows(const GsCtx<T>& x, const unsigned* d, const Cx<T>* w, int to) {
    if (x.cs == 1) return;
#pragma unroll
    for (int k = 0; k < KN; ++k) {
        if (d[k] & kGsUp) st<T>(x.vup, to * x.ss + (d[k] & 0xffff), w[k]);
        if (d[k] & kGsDn) st<T>(x.vdn, to * x.ss + (d[k] & 0xffff), w[k]);
    }
}
template <typename T, int KN>
__device__ __forceinline__ void take_rows(const GsCtx<T>& x, const unsigned* d, Cx<T>* w, int from) {
    if (x.cs == 1) return;
#pragma unroll
    for (int k = 0; k < KN; ++k)
        if (d[k] & kGsHalo) w[k] = ld<T>(x.V, from * x.ss + (d[k] & 0xffff));
}

// the warp's share of ||w||^2 on the own rows, as scalar q of the sums
template <typename T, int KN>
__device__ __forceinline__ void norm_share(const GsCtx<T>& x, const unsigned* d, const Cx<T>* w, int q) {
    T acc = T(0);
#pragma unroll
    for (int k = 0; k < KN; ++k) {
        const Cx<T> u = d[k] & kGsIn ? w[k] : cx<T>(0, 0);
        acc = fmaT(u.re, u.re, fmaT(u.im, u.im, acc));
    }
    __syncwarp();  // (a group of sums may have written there)
    warp_sums<T, 1>(&acc, &x.sh->red[threadIdx.x >> 5][q]);
}

// w orthogonalised against v_0..v_{nv-1} by classical Gram-Schmidt, twice: column nv - 1 of H; its
// squared norm the return value.  Straight-line over a thread's KN nodes (those it has not read an
// entry that is 0), in groups of kGroup vectors.
template <typename T, int KN>
__device__ __forceinline__ T orthogonalise(GsCtx<T>& x, const unsigned* d, Cx<T>* w, int nv, bool more) {
    constexpr int kGroup = 4;
    GsShared<T>& sh = *x.sh;
    T(*H)[kGsScal] = sh.H[(nv - 1) & 1], (*L)[kGsScal] = sh.L[(nv - 1) & 1];
    if (more) send_rows<T, KN>(x, d, w, nv);
    T sq = T(0);
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        const vec2<T>* v0 = x.V;
#pragma unroll 1
        for (int i0 = 0; i0 < nv; i0 += kGroup, v0 += kGroup * x.ss) {
            T acc[2 * kGroup];
#pragma unroll
            for (int i = 0; i < 2 * kGroup; ++i) acc[i] = T(0);
#pragma unroll
            for (int k = 0; k < KN; ++k) {
                const vec2<T>* p = v0 + (d[k] & 0xffff);
                const Cx<T> u = d[k] & kGsIn ? w[k] : cx<T>(0, 0);
#pragma unroll
                for (int i = 0; i < kGroup; ++i) {
                    const Cx<T> v = i0 + i < nv ? ld<T>(p, i * x.ss) : cx<T>(0, 0);
                    acc[2 * i] = fmaT(v.re, u.re, fmaT(v.im, u.im, acc[2 * i]));
                    acc[2 * i + 1] = fmaT(v.re, u.im, fmaT(-v.im, u.re, acc[2 * i + 1]));
                }
            }
            warp_sums<T, 2 * kGroup>(acc, &sh.red[threadIdx.x >> 5][2 * i0]);
        }
        if (pass) norm_share<T, KN>(x, d, w, 2 * nv);
        cluster_sums<T>(x, 2 * nv + pass, H[pass], L[pass], pass ? -1 : nv - 2);
        if (!pass && more) take_rows<T, KN>(x, d, w, nv);
        v0 = x.V;
#pragma unroll 1
        for (int i0 = 0; i0 < nv; i0 += kGroup, v0 += kGroup * x.ss) {
            Cx<T> c[kGroup];
#pragma unroll
            for (int i = 0; i < kGroup; ++i) {
                c[i] = i0 + i < nv ? cx<T>(-H[pass][2 * (i0 + i)], -H[pass][2 * (i0 + i) + 1]) : cx<T>(0, 0);
                if (pass) sq += c[i].re * c[i].re + c[i].im * c[i].im;
            }
#pragma unroll
            for (int k = 0; k < KN; ++k) {
                const vec2<T>* p = v0 + (d[k] & 0xffff);
#pragma unroll
                for (int i = 0; i < kGroup; ++i)
                    w[k] = fma_c(c[i], i0 + i < nv ? ld<T>(p, i * x.ss) : cx<T>(0, 0), w[k]);
            }
        }
    }
    const T before = H[1][2 * nv];
    if (sq <= before * T(1.0 / 64)) return before + (L[1][2 * nv] - sq);
    norm_share<T, KN>(x, d, w, 0);
    cluster_sums<T>(x, 1, &sh.tmp, &sh.low);
    return sh.tmp;
}

// grid (nb * cs), clusters of cs CTAs: problem blockIdx.x / cs.  x (in/out; xzero: from 0) and b at
// problem offsets pb * N.  KN: nodes a thread at most (own and halo rows).
template <typename T, int KN>
__global__ void __launch_bounds__(GsCfg<T>::kThreads) k_gs_step(const __grid_constant__ MArgs<T> a,
                                                                const vec2<T>* __restrict__ bvec, vec2<T>* xvec,
                                                                int xzero, int its, int cs) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int NT = blockDim.x;
    const int pb = blockIdx.x / cs;
    extern __shared__ __align__(128) unsigned char gs_smem[];
    GsShared<T>& sh = *reinterpret_cast<GsShared<T>*>(gs_smem);
    const int n = a.g.n, nn = a.g.nn, tid = threadIdx.x;
    GsCtx<T> X;
    X.sh = &sh;
    X.V = reinterpret_cast<vec2<T>*>(gs_smem + kGsHead<T>);
    X.rank = blockIdx.x - pb * cs;
    X.cs = cs;
    X.W = nn + 2;
    X.ss = ((nn + cs - 1) / cs + 2) * X.W;
    X.phase = 0;
    const int f0 = X.rank * nn / cs;
    X.R = (X.rank + 1) * nn / cs - f0;
    const int W = X.W, M = X.R * nn;
    const vec2<T>* bb = bvec + (long long)pb * a.g.N + (long long)f0 * nn;
    vec2<T>* xb = xvec + (long long)pb * a.g.N + (long long)f0 * nn;
    const bool has_up = X.rank > 0, has_dn = X.rank + 1 < cs;
    const int up = has_up ? nn : 0, dn = has_dn ? nn : 0;
    unsigned d[KN];
    Cx<T> w[KN];  // (b at first)
    auto dirichlet = [&](int i, int j) {
        return (i == 0 && a.g.dir[0]) || (i == n && a.g.dir[1]) || (j == 0 && a.g.dir[2]) || (j == n && a.g.dir[3]);
    };
    // what depends on nothing before this launch: node words, zeros beside the rows and in the rows
    // beyond the grid
    auto coords = [&](int q, int* i, int* j) {
        if (q < M) {
            const int r = q / nn;
            *i = q - r * nn;
            *j = f0 + r;
        } else {
            const bool above = q - M < up;
            *i = q - M - (above ? 0 : up);
            *j = above ? f0 - 1 : f0 + X.R;
        }
    };
#pragma unroll
    for (int k = 0; k < KN; ++k) {
        const int q = tid + k * NT;
        d[k] = 0;
        if (q < M + up + dn) {
            int i, j;
            coords(q, &i, &j);
            const int r = j - f0;
            const int tx = i == 0 ? 0 : (i == n ? 2 : 1), ty = j == 0 ? 0 : (j == n ? 2 : 1);
            d[k] = (unsigned)((r + 1) * W + i + 1);
            if (q < M)
                d[k] |= (unsigned)(tx == 1 && ty == 1 ? 8 : bclass2(tx, ty)) << 16 | (has_up && r == 0 ? kGsUp : 0) |
                        (has_dn && r == X.R - 1 ? kGsDn : 0) | (dirichlet(i, j) ? 0 : kGsFree) | kGsIn;
            else
                d[k] |= kGsHalo;
        }
        if (KN > 2 && __all_sync(0xffffffffu, (d[k] >> 16 & 15) == 8)) d[k] |= kGsInner;
    }
    {
        const int slots = max(its, 2), rows = X.R + 2;
        for (int t = tid; t < slots * rows; t += NT) {
            const int q = t / rows, r = t - q * rows;
            vec2<T>* row = X.V + q * X.ss + r * W;
            st<T>(row, 0, cx<T>(0, 0));
            st<T>(row, W - 1, cx<T>(0, 0));
        }
        for (int t = tid; t < W; t += NT)
            for (int q = 0; q < slots; ++q) {
                if (!has_up) st<T>(X.V, q * X.ss + t, cx<T>(0, 0));
                if (!has_dn) st<T>(X.V, q * X.ss + (X.R + 1) * W + t, cx<T>(0, 0));
            }
    }
    if (cs > 1) {
        cg::this_cluster().sync();  // every CTA is in place
        const int ru = has_up ? f0 - (X.rank - 1) * nn / cs : 0;  // rows of the CTA above
        X.vup = has_up ? cg::this_cluster().map_shared_rank(X.V, X.rank - 1) + ru * W : nullptr;
        X.vdn = has_dn ? cg::this_cluster().map_shared_rank(X.V, X.rank + 1) - X.R * W : nullptr;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (a.pc && problem_skipped(a, pb)) return;  // the whole cluster
    if (tid < 9) {
        const PCoef<T>& c = a.pc ? a.pc[pb] : a.c0;
        GsWeights<T>& k = sh.wt[tid];
        const bool in = tid == 8;
        k.w[0] = in ? c.iw[0] : c.bw[tid][0];
        k.w[1] = in ? c.iw[1] : c.bw[tid][1];
        k.w[2] = in ? c.iw[1] : c.bw[tid][2];
        k.w[3] = in ? c.iw[2] : c.bw[tid][3];
        k.dinv = in ? c.wdinv : c.bdinv[tid];
    }
    // b; x with its halo rows to basis vector 1 (first written when every CTA is past its use here)
#pragma unroll
    for (int k = 0; k < KN; ++k) {
        w[k] = d[k] & kGsFree ? ld<T>(bb, tid + k * NT) : cx<T>(0, 0);
        if (!xzero && d[k]) {
            int i, j;
            coords(tid + k * NT, &i, &j);
            st<T>(X.V, X.ss + (d[k] & 0xffff),
                  dirichlet(i, j) ? cx<T>(0, 0) : ld<T>(xb, (long long)(j - f0) * nn + i));
        }
    }
    __syncthreads();
    // z0 = omega D^{-1} (b - A x), beta = ||z0||, v_0 = z0 / beta; then w = omega D^{-1} A v_j
#pragma unroll 1
    for (int j = -1; j < its; ++j) {
        const bool more = j + 1 < its;
        T h2;
        // (keeps every node's addresses from being worked out before the loop, and spilled)
#pragma unroll
        for (int k = 0; k < KN; ++k) asm volatile("" : "+r"(d[k]));
        if (j >= 0 || !xzero) {
            const vec2<T>* f = X.V + (j < 0 ? 1 : j) * X.ss;
#pragma unroll
            for (int k = 0; k < KN; ++k) {
                // (a node without an unknown applies the stencil at a place where it can)
                Cx<T> dinv;
                const bool fr = d[k] & kGsFree;
                const Cx<T> ax = band_apply<T>(sh.wt, f, W, fr ? d[k] : (unsigned)(W + 1) | 8u << 16, &dinv);
                const Cx<T> v = cmul(dinv, j < 0 ? w[k] - ax : ax);
                w[k] = fr ? v : cx<T>(0, 0);
            }
        } else {
#pragma unroll
            for (int k = 0; k < KN; ++k)
                if (d[k] & kGsFree) w[k] = cmul(sh.wt[(d[k] >> 16) & 15].dinv, w[k]);
        }
        if (j >= 0) {
            h2 = orthogonalise<T, KN>(X, d, w, j + 1, more);
        } else {
            send_rows<T, KN>(X, d, w, 0);
            norm_share<T, KN>(X, d, w, 0);
            cluster_sums<T>(X, 1, &sh.beta2, &sh.low);
            take_rows<T, KN>(X, d, w, 0);
            h2 = sh.beta2;
        }
        const T h = sqrt(h2);
        if (tid == 0) {
            if (j >= 0)
                sh.h[j] = h;
            else
                sh.g[0] = cx<T>(h, 0);
        }
        if (!more) break;
        const T s = h > T(0) ? T(1) / h : T(0);
        vec2<T>* vn = X.V + (j + 1) * X.ss;
#pragma unroll
        for (int k = 0; k < KN; ++k)
            if (d[k]) st<T>(vn, d[k] & 0xffff, cx<T>(w[k].re * s, w[k].im * s));
        __syncthreads();
    }
    // x early: its latency runs beside the small problem
#pragma unroll
    for (int k = 0; k < KN; ++k) w[k] = !xzero && (d[k] & kGsIn) ? ld<T>(xb, tid + k * NT) : cx<T>(0, 0);
    if (tid < 32) {
        rotate_column<T>(sh, its - 1);
        __syncwarp();
        back_substitute<T>(sh, its);
    }
    __syncthreads();
    for (int i = 0; i < its; ++i) {
        const Cx<T> y = sh.ys[i];
#pragma unroll
        for (int k = 0; k < KN; ++k) w[k] = fma_c(y, ld<T>(X.V, i * X.ss + (d[k] & 0xffff)), w[k]);
    }
#pragma unroll
    for (int k = 0; k < KN; ++k)
        if (d[k] & kGsIn) st<T>(xb, tid + k * NT, w[k]);
}

template <typename T, int KN>
int gs_cluster_of() {
    if (cudaFuncSetAttribute(k_gs_step<T, KN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGsSmemMax) !=
        cudaSuccess)
        return -1;
    cudaFuncSetAttribute(k_gs_step<T, KN>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (int cs = kGsClusterMax; cs > 1; cs >>= 1) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)cs);
        cfg.blockDim = dim3(GsCfg<T>::kThreads);
        cfg.dynamicSmemBytes = kGsSmemMax;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)cs;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int active = 0;
        if (cudaOccupancyMaxActiveClusters(&active, k_gs_step<T, KN>, &cfg) == cudaSuccess && active >= 1) return cs;
    }
    return 1;
}

// Configure k_gs_step<T> and find the largest cluster of it that the device holds (once per device; asked
// for at every smoothing step, so the answer is read without the lock).
template <typename T>
int gs_cluster_max() {
    constexpr int kMaxDev = 64;
    static std::mutex mu;
    static std::atomic<int> held[kMaxDev];  // 0: not looked at yet, -1: not available
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
        cudaGetLastError();
        return -1;
    }
    int cs = held[dev].load(std::memory_order_acquire);
    if (cs) return cs;
    std::lock_guard<std::mutex> g(mu);
    cs = held[dev].load(std::memory_order_relaxed);
    if (!cs) {
        cs = std::min({gs_cluster_of<T, 1>(), gs_cluster_of<T, 2>(), gs_cluster_of<T, 5>()});
        cudaGetLastError();
        held[dev].store(cs, std::memory_order_release);
    }
    return cs;
}

// nodes of the largest band with its halo rows
inline long long gs_band(int nn, int cs) { return (long long)((nn + cs - 1) / cs + (cs > 1 ? 2 : 0)) * nn; }

template <typename T>
size_t gs_step_smem(int nn, int its, int cs) {
    const size_t rows = (size_t)(nn + cs - 1) / cs;
    return kGsHead<T> + (size_t)std::max(its, 2) * (rows + 2) * (nn + 2) * sizeof(vec2<T>);
}

}  // namespace

template <typename T>
int gs_step_cluster(const GridDesc& g, int its) {
    if (g.dim != 2 || its < 1 || its > kGsMaxIts) return 0;
    const int most = gs_cluster_max<T>();
    int best = 0;
    for (int cs = 1; cs <= most && cs <= g.nn; cs <<= 1) {
        const long long nodes = gs_band(g.nn, cs);
        if (nodes > 5LL * GsCfg<T>::kThreads || gs_step_smem<T>(g.nn, its, cs) > kGsSmemMax) continue;
        best = cs;
        if (nodes <= kGsBand) break;
    }
    return best;
}

template <typename T>
cudaError_t launch_gs_step(const MArgs<T>& a, const vec2<T>* b, vec2<T>* x, int xzero, int its, int cs,
                           cudaStream_t s) {
    if (cs < 1 || (!a.pc && a.nb != 1)) return cudaErrorInvalidValue;
    const long long nodes = gs_band(a.g.nn, cs);
    // complex64: a warp per scalar of a sum at least, for the sums over the warps are a serial chain
    // (751 -> 712 us with the set-up before the wait for the previous kernel); complex128: as few as the
    // nodes need, for each costs the FP64 pipe its time
    const int most = GsCfg<T>::kThreads;
    const int least = sizeof(T) == 8 ? 64 : std::min(most, 32 * (2 * its + 1));
    const int kn = nodes <= most ? 1 : nodes <= 2 * most ? 2 : 5;
    const dim3 grd((unsigned)(a.nb * cs));
    const dim3 blk((unsigned)std::max((long long)least, ((nodes + kn - 1) / kn + 31) / 32 * 32));
    const size_t sm = gs_step_smem<T>(a.g.nn, its, cs);
    if (kn == 1) return klaunch(k_gs_step<T, 1>, grd, blk, sm, s, cs, a, b, x, xzero, its, cs);
    if (kn == 2) return klaunch(k_gs_step<T, 2>, grd, blk, sm, s, cs, a, b, x, xzero, its, cs);
    return klaunch(k_gs_step<T, 5>, grd, blk, sm, s, cs, a, b, x, xzero, its, cs);
}

template <typename T>
cudaError_t launch_gs_dot(const vec2<T>* V, long long ldv, int nv, const vec2<T>* w, long long N, double2* part,
                          const Batch& bt, cudaStream_t s) {
    if (nv < 1 || nv > kGsMaxVec) return cudaErrorInvalidValue;
    const dim3 grd((unsigned)gs_blocks(N), (unsigned)bt.nb);
    return klaunch(k_gs_dot<T>, grd, dim3(kGsThreads), 0, s, 1, V, ldv, nv, w, N, part, bt);
}

template <typename T>
cudaError_t launch_gs_orth(vec2<T>* w, const vec2<T>* V, long long ld, int nv, long long N, const double2* part,
                           double2* ls, int col, int accumulate, double2* part2, const Batch& bt, cudaStream_t s) {
    if (nv < 1 || nv > kGsMaxVec || col < 0 || col >= kGsMaxIts) return cudaErrorInvalidValue;
    const dim3 grd((unsigned)gs_blocks(N), (unsigned)bt.nb);
    return klaunch(k_gs_orth<T>, grd, dim3(kGsThreads), 0, s, 1, w, V, ld, nv, N, part, ls, col, accumulate, part2,
                   bt);
}

template <typename T>
cudaError_t launch_gs_scale(vec2<T>* out, const vec2<T>* w, long long N, const double2* part2, double2* ls, int col,
                            const Batch& bt, cudaStream_t s) {
    if (col >= kGsMaxIts) return cudaErrorInvalidValue;
    const int nblk = gs_blocks(N);
    const dim3 grd((unsigned)nblk, (unsigned)bt.nb);
    return klaunch(k_gs_scale<T>, grd, dim3(kGsThreads), 0, s, 1, out, w, N, part2, nblk, ls, col, bt);
}

template <typename T>
cudaError_t launch_gs_update(vec2<T>* x, const vec2<T>* V, long long ld, int m, long long N, const double2* ls,
                             int overwrite, const Batch& bt, cudaStream_t s) {
    if (m < 1 || m > kGsMaxIts) return cudaErrorInvalidValue;
    const dim3 grd((unsigned)gs_blocks(N), (unsigned)bt.nb);
    return klaunch(k_gs_update<T>, grd, dim3(kGsThreads), 0, s, 1, x, V, ld, m, N, ls, overwrite, bt);
}

#define HH_GS_INST(T)                                                                                                 \
    template cudaError_t launch_gs_dot<T>(const vec2<T>*, long long, int, const vec2<T>*, long long, double2*,        \
                                          const Batch&, cudaStream_t);                                                \
    template cudaError_t launch_gs_orth<T>(vec2<T>*, const vec2<T>*, long long, int, long long, const double2*,       \
                                           double2*, int, int, double2*, const Batch&, cudaStream_t);                 \
    template cudaError_t launch_gs_scale<T>(vec2<T>*, const vec2<T>*, long long, const double2*, double2*, int,       \
                                            const Batch&, cudaStream_t);                                              \
    template cudaError_t launch_gs_update<T>(vec2<T>*, const vec2<T>*, long long, int, long long, const double2*,     \
                                             int, const Batch&, cudaStream_t);
template int gs_step_cluster<float>(const GridDesc&, int);
template int gs_step_cluster<double>(const GridDesc&, int);
template cudaError_t launch_gs_step<float>(const MArgs<float>&, const vec2<float>*, vec2<float>*, int, int, int,
                                           cudaStream_t);
template cudaError_t launch_gs_step<double>(const MArgs<double>&, const vec2<double>*, vec2<double>*, int, int, int,
                                            cudaStream_t);
HH_GS_INST(float)
HH_GS_INST(double)
#undef HH_GS_INST

}  // namespace hh
