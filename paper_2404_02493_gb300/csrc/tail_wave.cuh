// Shared-memory tail of the wave cycle (Algorithm 1 on the levels below the
// ADR corrections).
//
// On the small wave levels every Chebyshev step (eq. cheb) is a launch of its
// own and costs more than its work.  For an instance whose levels l0 .. L-1
// (l0 >= 4, all smoothed) are small enough, the sub-cycle wave(l0 .. L) runs
// as three launches:
//
//   k_wave_down  one block of WT_THREADS per instance; for l = l0 .. L-1: q
//                Chebyshev steps from x = 0 on the level's g, x to its SU
//                slot, the residual g - A x restricted by full weighting to
//                the SG slot of level l+1 (the coarsest one included)
//   k_coarse     the coarsest solve of the multi-launch path
//   k_wave_up    one block per instance; for l = L-1 .. l0: x' = x + P e
//                (e the result of level l+1), q Chebyshev steps from x', the
//                result to the level's SU slot
//
// What bounds it: 20 dependent stencil passes per level in one block, each its
// SM's shared-memory traffic and a barrier.  A thread owns wt_rpt() rows of a
// column: x, d, g and the diagonal of its nodes stay in registers, north and
// south neighbours inside its rows too, and the two shared vectors (x, the
// residual t) have a zero border, so a pass loads 2.5 values per node and
// stores one.  With every operand in shared memory, a test per neighbour, the
// step coefficients read from global memory inside the chain and the level
// chain followed pointer by pointer the two launches took 29 and 26 us for
// levels of 63 and 31; now 21 and 19 us (of which ~5 are the launch and the first loads).
//
// In FP64 the four rows a thread would need for 64 rows do not fit its
// registers (a complex value takes four), so a level of more than 32 rows keeps
// its launches, which also spread the FP64 work over all SMs: with a tail that
// took levels up to 51 x 51 in shared memory an FGMRES step without ADR
// corrections ran 702 us at n = 264 (level of 33), 917 at n = 400 (50), 1277 at n =
// 700 (43), with those levels per launch 592, 695 and 1107 us.
//
// Slots are those of the multi-launch path (k_cheb_step, k_restrict<MODE_HELM>,
// k_prolong<PMODE_ADD>) and in FP64 its per-node arithmetic; in FP32 the
// Laplacian is a sum of differences (wave_nodes.cuh).  The Chebyshev
// direction lives in registers only (the first step of a smoothing does not
// read it).  Only block barriers are used; every thread runs the same level
// loop.
#pragma once
#include "wave_nodes.cuh"

namespace wadr {

constexpr int TS_MAXL = 8;    // levels of a chain, the coarsest included
template <typename T> __host__ __device__ constexpr int wt_maxny() { return WT_THREADS / WT_MAXN * wt_rpt<T>(); }

// dynamic shared memory for a first level of n x ny nodes: x and t with a
// zero border, and the next level's vector (right-hand side going down,
// solution with a zero border coming up)
template <typename T> __host__ __device__ constexpr long long wt_smem(int n, int ny) {
    return (long long)sizeof(cplx<T>) * (2LL * (n + 2) * (ny + 2) + (long long)(n / 2 + 2) * (ny / 2 + 2));
}

// The level chain of this block's instance (TS_MAXL descriptor indices, -1
// after the coarsest), its descriptors and Chebyshev coefficients in shared
// memory; returns the number of levels.
template <typename T>
__device__ __forceinline__ int wt_chain(const LevelDesc* __restrict__ D, const int* __restrict__ chain, LevelDesc* Lv,
                                        int* didx, T (*cc)[2][16]) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid < TS_MAXL) didx[tid] = chain[blockIdx.x * TS_MAXL + tid];
    __syncthreads();
    int nl = 0;
    while (nl < TS_MAXL && didx[nl] >= 0) ++nl;
    for (int k = w; k < nl; k += WT_THREADS / 32) copy_desc(Lv[k], D + didx[k], lane);
    __syncthreads();
    for (int e = tid; e < nl * 32; e += WT_THREADS) {
        const int k = e >> 5, c = (e >> 4) & 1, m = e & 15;
        cc[k][c][m] = scalp<T>(Lv[k])[(c ? S::CHEB_C2 : S::CHEB_C1) + m];
    }
    __syncthreads();
    return nl;
}

// zero the borders (and everything else) of the two shared vectors of a level
template <typename T> __device__ __forceinline__ void wt_zero(cplx<T>* X, cplx<T>* Tt, const LevelDesc& d) {
    const int e = (d.n + 2) * (d.ny + 2);
    for (int q = threadIdx.x; q < e; q += WT_THREADS) X[q] = Tt[q] = zero2<T>();
}

// ------------------------------------------------------------ down
template <typename T>
__global__ void __launch_bounds__(WT_THREADS, 1) k_wave_down(const LevelDesc* __restrict__ D,
                                                             const int* __restrict__ chain, int q) {
    extern __shared__ __align__(16) unsigned char wt_smem_raw[];
    __shared__ LevelDesc Lv[TS_MAXL];
    __shared__ int didx[TS_MAXL];
    __shared__ T cc[TS_MAXL][2][16];
    const int nl = wt_chain<T>(D, chain, Lv, didx, cc);
    const int E0 = (Lv[0].n + 2) * (Lv[0].ny + 2);
    cplx<T>* const X = reinterpret_cast<cplx<T>*>(wt_smem_raw);
    cplx<T>* const Tt = X + E0;
    cplx<T>* const Gn = Tt + E0;       // the next level's right-hand side
    constexpr int RPT = WtNodes<T>::RPT;
    for (int k = 0; k + 1 < nl; ++k) {
        const LevelDesc& d = Lv[k];
        const LevelDesc& dc = Lv[k + 1];
        const T ih2 = LC<T>::ih2(d);
        WtNodes<T> N;
        N.place(d.n, d.n, d.ny);
        const cplx<T>* gg = slot<T>(d, SG);
#pragma unroll
        for (int r = 0; r < RPT; ++r)
            if (N.in[r]) {
                N.g[r] = k == 0 ? gg[(long long)(N.j0 + r) * d.pitch + N.i] : Gn[(N.j0 + r) * d.n + N.i];
                N.dg[r] = wt_diag<T>(d, N.i, N.j0 + r);
            }
        wt_zero<T>(X, Tt, d);
        __syncthreads();
        wt_cheb<T>(N, q, true, X, Tt, ih2, cc[k]);
        // x to SU; r = g - A x
        cplx<T>* xs = slot<T>(d, SU);
        cplx<T> t[RPT];
#pragma unroll
        for (int r = 0; r < RPT; ++r)
            if (N.in[r]) xs[(long long)(N.j0 + r) * d.pitch + N.i] = N.x[r];
        N.residual(t, X, Tt, ih2, false);
        __syncthreads();
        // full weighting (1/16)[1 2 1; 2 4 2; 1 2 1] of r; coarse node I on fine node 2I+1
        const int nc = dc.n, ncy = dc.ny, W = N.W;
        cplx<T>* gc = slot<T>(dc, SG);
        for (int J = threadIdx.x / WT_MAXN, I = N.i; J < ncy; J += WT_THREADS / WT_MAXN)
            if (I < nc) {
                const cplx<T>* b = Tt + (2 * J + 2) * W + 2 * I + 2;
                const cplx<T> s2 = cadd<T>(cadd<T>(b[-1], b[1]), cadd<T>(b[-W], b[W]));
                const cplx<T> s1 = cadd<T>(cadd<T>(b[-W - 1], b[-W + 1]), cadd<T>(b[W - 1], b[W + 1]));
                const cplx<T> v = cscale<T>(cadd<T>(cadd<T>(cscale<T>(b[0], T(4)), cscale<T>(s2, T(2))), s1), T(0.0625));
                Gn[J * nc + I] = v;
                gc[(long long)J * dc.pitch + I] = v;
            }
        __syncthreads();
    }
}

// ------------------------------------------------------------ up
template <typename T>
__global__ void __launch_bounds__(WT_THREADS, 1) k_wave_up(const LevelDesc* __restrict__ D,
                                                           const int* __restrict__ chain, int q) {
    extern __shared__ __align__(16) unsigned char wt_smem_raw[];
    __shared__ LevelDesc Lv[TS_MAXL];
    __shared__ int didx[TS_MAXL];
    __shared__ T cc[TS_MAXL][2][16];
    const int nl = wt_chain<T>(D, chain, Lv, didx, cc);
    const int E0 = (Lv[0].n + 2) * (Lv[0].ny + 2);
    cplx<T>* const X = reinterpret_cast<cplx<T>*>(wt_smem_raw);
    cplx<T>* const Tt = X + E0;
    cplx<T>* const E = Tt + E0;        // solution of the next coarser level, zero border
    constexpr int RPT = WtNodes<T>::RPT;
    for (int e = threadIdx.x; e < (Lv[0].n / 2 + 2) * (Lv[0].ny / 2 + 2); e += WT_THREADS) E[e] = zero2<T>();
    __syncthreads();
    {
        const LevelDesc& dL = Lv[nl - 1];
        const cplx<T>* xg = slot<T>(dL, SU);
        for (int J = threadIdx.x / WT_MAXN, I = threadIdx.x & (WT_MAXN - 1); J < dL.ny; J += WT_THREADS / WT_MAXN)
            if (I < dL.n) E[(J + 1) * (dL.n + 2) + I + 1] = xg[(long long)J * dL.pitch + I];
    }
    for (int k = nl - 2; k >= 0; --k) {
        const LevelDesc& d = Lv[k];
        const int Wc = Lv[k + 1].n + 2;
        const T ih2 = LC<T>::ih2(d);
        WtNodes<T> N;
        N.place(d.n, d.n, d.ny);
        const cplx<T>* xg = slot<T>(d, SU);
        const cplx<T>* gg = slot<T>(d, SG);
#pragma unroll
        for (int r = 0; r < RPT; ++r)
            if (N.in[r]) {
                const long long p = (long long)(N.j0 + r) * d.pitch + N.i;
                N.x[r] = xg[p];
                N.g[r] = gg[p];
                N.dg[r] = wt_diag<T>(d, N.i, N.j0 + r);
            }
        wt_zero<T>(X, Tt, d);
        __syncthreads();
        // x' = x + P e (bilinear; coarse node I on fine node 2I+1)
#pragma unroll
        for (int r = 0; r < RPT; ++r)
            if (N.in[r]) {
                const int i = N.i, j = N.j0 + r, ia = (i - 1) >> 1, ja = (j - 1) >> 1;
                const T wa0 = (i & 1) ? T(1) : T(0.5), wa1 = T(1) - wa0;
                const T wb0 = (j & 1) ? T(1) : T(0.5), wb1 = T(1) - wb0;
                const cplx<T>* e = E + (ja + 1) * Wc + ia + 1;
                cplx<T> v = cscale<T>(cadd<T>(cscale<T>(e[0], wa0), cscale<T>(e[1], wa1)), wb0);
                v = cadd<T>(v, cscale<T>(cadd<T>(cscale<T>(e[Wc], wa0), cscale<T>(e[Wc + 1], wa1)), wb1));
                N.x[r] = cadd<T>(N.x[r], v);
                X[N.at(r)] = N.x[r];
            }
        __syncthreads();
        wt_cheb<T>(N, q, false, X, Tt, ih2, cc[k]);
        cplx<T>* xs = slot<T>(d, SU);
#pragma unroll
        for (int r = 0; r < RPT; ++r)
            if (N.in[r]) xs[(long long)(N.j0 + r) * d.pitch + N.i] = N.x[r];
        if (k > 0) {
            const int e = (d.n + 2) * (d.ny + 2);
            for (int p = threadIdx.x; p < e; p += WT_THREADS) E[p] = X[p];   // borders zero as in X
            __syncthreads();
        }
    }
}

}  // namespace wadr
