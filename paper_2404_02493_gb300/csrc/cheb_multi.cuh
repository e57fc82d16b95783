// All q Chebyshev steps of one smoothing (eq. cheb) in one launch, for the
// small wave levels (temporal blocking), complex FP32.
//
// A level of a few hundred thousand points gives a one-step launch too
// little work per block to hide its own latency (load, two stencil passes,
// store), so q steps cost q such latencies.  Here a block loads an output
// tile of TS x TS nodes with a ring of H = 2q nodes (x unless it is zero, g,
// and the Helmholtz diagonal formed from k and the sponge term) into shared
// memory and runs the q steps there: step m forms t = g - A x on the ring of
// width H - 2m - 1 around the tile, then s = A^* t, d <- c1[m] d + c2[m] s,
// x <- x + d on the ring of width H - 2m - 2.  The last step leaves x valid on
// the tile itself, which is written to slot sxout (!= sxin: other blocks read
// the input on their rings).  d starts at zero (c1[0] = 0) and never leaves
// shared memory.  Nodes outside the grid hold zero, as in k_cheb_step; the
// arithmetic per node and its order are those of k_cheb_step.
#pragma once
#include "wave_nodes.cuh"

namespace wadr {

// shared memory of a block: x, d, t, g and the diagonal on (TS + 2H)^2 nodes
template <typename T> __host__ __device__ constexpr int cm_smem(int TS, int q) {
    return 5 * (TS + 4 * q) * (TS + 4 * q) * (int)sizeof(cplx<T>);
}

template <typename T, int TS>
__global__ void __launch_bounds__(NT) k_cheb_multi(const __grid_constant__ KDesc A, const Seg* __restrict__ Sg,
                                                   int nseg, int sxin, int sxout, int q, int xzero) {
    extern __shared__ __align__(16) unsigned char cm_smem_[];
    __shared__ LevelDesc d;
    SegCtx c = seg_begin(A, Sg, nseg, d);
    const int H = 2 * q, W = TS + 2 * H, WW = W * W;
    cplx<T>* const X = reinterpret_cast<cplx<T>*>(cm_smem_);
    cplx<T>* const D = X + WW;
    cplx<T>* const Tt = D + WW;
    cplx<T>* const G = Tt + WW;
    cplx<T>* const DG = G + WW;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + ty * blockDim.x;
    const int n = d.n, ny = d.ny, pitch = d.pitch;
    const int ntx = (n + TS - 1) / TS, ntiles = ntx * ((ny + TS - 1) / TS);
    const cplx<T>* const xin = slot<T>(d, sxin);
    const cplx<T>* const gv = slot<T>(d, SG);
    cplx<T>* const xout = slot<T>(d, sxout);
    const T* const kf = reinterpret_cast<const T*>(d.kf);
    const T* const sgf = reinterpret_cast<const T*>(d.sig);
    const T ih2 = LC<T>::ih2(d);
    const T* const scl = scalp<T>(d);
    for (int t = c.lb; t < ntiles; t += c.nb) {
        const int x0 = (t % ntx) * TS - H, y0 = (t / ntx) * TS - H;   // grid node of region node (0, 0)
        // load the region; zero outside the grid
        for (int e = tid; e < WW; e += NT) {
            const int r = e / W, cc = e - r * W;
            const int gi = x0 + cc, gj = y0 + r;
            cplx<T> xv = zero2<T>(), gval = zero2<T>(), dg = zero2<T>();
            if ((unsigned)gi < (unsigned)n && (unsigned)gj < (unsigned)ny) {
                const long long p = (long long)gj * pitch + gi;
                if (!xzero) xv = xin[p];
                gval = gv[p];
                dg = helm_diag_h2<T>(d, gi, gj, kf[p], sgf ? sgf[p] : T(0));
            }
            X[e] = xv;
            D[e] = zero2<T>();
            G[e] = gval;
            DG[e] = dg;
        }
        __syncthreads();
        for (int m = 0; m < q; ++m) {
            // t = g - A x on rows / columns [lo, W - lo)
            const int lo = 2 * m + 1;
            const bool xz = xzero && m == 0;
            for (int r = lo + ty; r < W - lo; r += BY)
                for (int cc = lo + tx; cc < W - lo; cc += BX) {
                    const int e = r * W + cc;
                    const int gi = x0 + cc, gj = y0 + r;
                    cplx<T> tv = zero2<T>();
                    if ((unsigned)gi < (unsigned)n && (unsigned)gj < (unsigned)ny) {
                        tv = G[e];
                        if (!xz) {
                            const cplx<T> sn = cadd<T>(cadd<T>(X[e - 1], X[e + 1]), cadd<T>(X[e - W], X[e + W]));
                            tv = csub<T>(tv, cscale<T>(csub<T>(cmul<T>(DG[e], X[e]), sn), ih2));
                        }
                    }
                    Tt[e] = tv;
                }
            __syncthreads();
            // s = A^* t; d = c1 d + c2 s; x += d on [lo + 1, W - lo - 1)
            const T c1 = scl[S::CHEB_C1 + m], c2 = scl[S::CHEB_C2 + m];
            const int lo2 = lo + 1;
            for (int r = lo2 + ty; r < W - lo2; r += BY)
                for (int cc = lo2 + tx; cc < W - lo2; cc += BX) {
                    const int e = r * W + cc;
                    const int gi = x0 + cc, gj = y0 + r;
                    if ((unsigned)gi < (unsigned)n && (unsigned)gj < (unsigned)ny) {
                        const cplx<T> sn =
                            cadd<T>(cadd<T>(Tt[e - 1], Tt[e + 1]), cadd<T>(Tt[e - W], Tt[e + W]));
                        cplx<T> dg = DG[e];
                        dg.y = -dg.y;
                        const cplx<T> sv = cscale<T>(csub<T>(cmul<T>(dg, Tt[e]), sn), ih2);
                        cplx<T> dn = cscale<T>(sv, c2);
                        if (c1 != T(0)) dn = cadd<T>(dn, cscale<T>(D[e], c1));
                        D[e] = dn;
                        X[e] = cadd<T>(xz ? zero2<T>() : X[e], dn);
                    }
                }
            __syncthreads();
        }
        // x on the tile
        for (int r = H + ty; r < H + TS; r += BY)
            for (int cc = H + tx; cc < H + TS; cc += BX) {
                const int gi = x0 + cc, gj = y0 + r;
                if (gi < n && gj < ny) xout[(long long)gj * pitch + gi] = X[r * W + cc];
            }
        __syncthreads();
    }
}

// The same smoothing with the region in registers and the Laplacian as a sum of
// differences (wave_nodes.cuh): a block of 1024 threads holds 64 columns of 16
// RPT rows, of which all but 2q on each side are its output tile (values on the outer ring go wrong by one node per
// stencil).  With every operand in shared memory, an in-grid test per node and
// stage and 256 threads per region, k_cheb_multi is bound by issue slots and
// barriers; here a stage is bound by its shared-memory loads, so that two rows
// per thread are the faster form while their tiles fit the SMs, and four
// (which recompute less) above.  q = 5: n = 511 24 us there, 13.3 here, n =
// 255 12.6 and 7.0, n = 127 9.2 and 7.3.  k_cheb_multi remains for
// longer smoothings, whose ring would leave too small a tile.
constexpr int CR_W = 64, CR_MAXQ = 8;
template <typename T, int RPT> __host__ __device__ constexpr int cr_smem() {
    return 2 * (CR_W + 2) * (CR_W / 4 * RPT + 2) * (int)sizeof(cplx<T>);
}
template <typename T, int RPT>
__global__ void __launch_bounds__(WT_THREADS, 1) k_cheb_region(const __grid_constant__ KDesc A,
                                                               const Seg* __restrict__ Sg, int nseg, int sxin,
                                                               int sxout, int q, int xzero) {
    constexpr int RH = WT_THREADS / WT_MAXN * RPT, NE = (CR_W + 2) * (RH + 2);
    static_assert(RH == CR_W / 4 * RPT && WT_MAXN == CR_W, "region");
    extern __shared__ __align__(16) unsigned char cr_smem_[];
    __shared__ LevelDesc d;
    __shared__ T cc[2][16];
    SegCtx c = seg_begin(A, Sg, nseg, d);
    cplx<T>* const X = reinterpret_cast<cplx<T>*>(cr_smem_);
    cplx<T>* const Tt = X + NE;
    const int tid = threadIdx.x, H = 2 * q, TX = CR_W - 2 * H, TY = RH - 2 * H;
    const int n = d.n, ny = d.ny, pitch = d.pitch;
    const int ntx = (n + TX - 1) / TX, ntiles = ntx * ((ny + TY - 1) / TY);
    const cplx<T>* const xin = slot<T>(d, sxin);
    const cplx<T>* const gv = slot<T>(d, SG);
    cplx<T>* const xout = slot<T>(d, sxout);
    const T ih2 = LC<T>::ih2(d);
    if (tid < 32) cc[tid >> 4][tid & 15] = scalp<T>(d)[((tid >> 4) ? S::CHEB_C2 : S::CHEB_C1) + (tid & 15)];
    for (int e = tid; e < NE; e += WT_THREADS) X[e] = Tt[e] = zero2<T>();
    __syncthreads();
    for (int t = c.lb; t < ntiles; t += c.nb) {
        const int x0 = (t % ntx) * TX - H, y0 = (t / ntx) * TY - H;
        WtNodes<T, RPT> N;
        N.place(CR_W, n, ny, x0, y0);
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            if (N.in[r]) {
                const int gi = x0 + N.i, gj = y0 + N.j0 + r;
                const long long p = (long long)gj * pitch + gi;
                if (!xzero) N.x[r] = xin[p];
                N.g[r] = gv[p];
                N.dg[r] = wt_diag<T>(d, gi, gj);
            }
            // (nodes outside the grid are zero in both vectors)
            X[N.at(r)] = N.x[r];
            Tt[N.at(r)] = zero2<T>();
        }
        __syncthreads();
        wt_cheb<T>(N, q, xzero, X, Tt, ih2, cc);
        if (N.i >= H && N.i < CR_W - H)
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                const int j = N.j0 + r;
                if (N.in[r] && j >= H && j < RH - H) xout[(long long)(y0 + j) * pitch + x0 + N.i] = N.x[r];
            }
        __syncthreads();
    }
}

}  // namespace wadr
