// Chebyshev steps (eq. cheb) of a block that holds a level, or a region of
// one, in registers and shared memory: used by the shared-memory tail of the
// wave cycle and by the one-launch smoothing of the small levels.
//
// A thread owns a few rows of a column; x, d, g and the diagonal of its nodes
// stay in registers, north and south neighbours inside its rows too, and the
// two shared vectors (x, the residual t) have a zero border, so a stencil
// pass loads 2.5 values per node (4 rows per thread) and stores one.
// In FP32 the Laplacian is a sum of differences: largest error of a cycle
// against 64 bits over media of n = 100 to 700 9.7e-7 -> 4.1e-7, residual after
// 20 steps with M = 8 at n = 511 off by 1e-6 (median) instead of 2e-6, for 2 us
// of the cycle at n = 127 (98 us) and 9 us at n = 1024 (393 us).
#pragma once
#include "kernels.cuh"

namespace wadr {

constexpr int WT_THREADS = 1024;
constexpr int WT_MAXN = 64;   // columns; nodes map to threads as 64 columns x 16 groups of rows
// rows per thread (64 registers a thread at 1024 threads)
template <typename T> __host__ __device__ constexpr int wt_rpt() { return sizeof(T) == 4 ? 4 : 2; }

// One thread's nodes of a level: rows j0 .. j0 + RPT - 1 of column i.
template <typename T, int RPT_ = wt_rpt<T>()> struct WtNodes {
    static constexpr int RPT = RPT_;
    cplx<T> x[RPT], g[RPT], dg[RPT];
    int i, j0, W;
    bool in[RPT];
    // the vectors hold w columns and a border; column 0, row 0 of them is node
    // (x0, y0) of a level of ny rows of n
    __device__ __forceinline__ void place(int w, int n, int ny, int x0 = 0, int y0 = 0) {
        i = threadIdx.x & (WT_MAXN - 1);
        j0 = (threadIdx.x / WT_MAXN) * RPT;
        W = w + 2;
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            in[r] = (unsigned)(x0 + i) < (unsigned)n && (unsigned)(y0 + j0 + r) < (unsigned)ny;
            x[r] = g[r] = dg[r] = zero2<T>();
        }
    }
    __device__ __forceinline__ int at(int r) const { return (j0 + r + 1) * W + i + 1; }
    // What dg v_r lacks of h^2 A v at row r (own rows in v, the others in V).
    // FP32: 4 v_r less the neighbours as a sum of differences (see helm_diff),
    // dg the rest of the diagonal; FP64: minus the neighbours, dg the whole.
    __device__ __forceinline__ cplx<T> lap(const cplx<T> (&v)[RPT], const cplx<T>* V, int r) const {
        const int p = at(r);
        const cplx<T> s = r > 0 ? v[r > 0 ? r - 1 : 0] : V[p - W];
        const cplx<T> n = r < RPT - 1 ? v[r < RPT - 1 ? r + 1 : 0] : V[p + W];
        if (sizeof(T) == 8) {
            const cplx<T> a = cadd<T>(cadd<T>(V[p - 1], V[p + 1]), cadd<T>(s, n));
            return mk<T>(-a.x, -a.y);
        }
        return cadd<T>(cadd<T>(csub<T>(v[r], V[p - 1]), csub<T>(v[r], V[p + 1])),
                       cadd<T>(csub<T>(v[r], s), csub<T>(v[r], n)));
    }
    // t = g - A x, to the shared vector Tt
    __device__ __forceinline__ void residual(cplx<T> (&t)[RPT], const cplx<T>* X, cplx<T>* Tt, T ih2, bool xz) const {
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            t[r] = g[r];
            if (!xz && in[r]) t[r] = csub<T>(g[r], cscale<T>(cfma<T>(dg[r], x[r], lap(x, X, r)), ih2));
            if (in[r]) Tt[at(r)] = t[r];
        }
    }
};

template <typename T> __device__ __forceinline__ cplx<T> wt_diag(const LevelDesc& d, int i, int j) {
    if (sizeof(T) == 8) return helm_diag_at<T>(d, i, j);
    return helm_diag4<T>(d, i, j, load_k<T>(d, i, j), load_sig<T>(d, i, j));
}

// q Chebyshev steps on a level: s = A^H t, t = g - A x; d = c2[m] s + c1[m] d
// (c1[0] = 0); x += d.  x of the nodes in registers and (unless xzero) in X.
template <typename T, int RPT>
__device__ __forceinline__ void wt_cheb(WtNodes<T, RPT>& N, int q, bool xzero, cplx<T>* X, cplx<T>* Tt, T ih2,
                                        const T (*c)[16]) {
    cplx<T> d[RPT], t[RPT];
#pragma unroll
    for (int r = 0; r < RPT; ++r) d[r] = zero2<T>();
    for (int m = 0; m < q; ++m) {
        N.residual(t, X, Tt, ih2, xzero && m == 0);
        __syncthreads();
        const T c1 = c[0][m], c2 = c[1][m];
#pragma unroll
        for (int r = 0; r < RPT; ++r)
            if (N.in[r]) {
                cplx<T> dg = N.dg[r];
                dg.y = -dg.y;
                const cplx<T> sv = cscale<T>(cfma<T>(dg, t[r], N.lap(t, Tt, r)), ih2);
                cplx<T> dn = cscale<T>(sv, c2);
                if (c1 != T(0)) dn = cadd<T>(dn, cscale<T>(d[r], c1));
                d[r] = dn;
                N.x[r] = cadd<T>(N.x[r], dn);
                X[N.at(r)] = N.x[r];
            }
        __syncthreads();
    }
}

}  // namespace wadr
