// Coarse part of the ADR V-cycle (Section 3.2.2) in one launch: a cluster of
// CS blocks per instance holds levels l0 .. L in distributed shared memory.
//
// What bounds these levels is not data (a few hundred KB) but the chain of
// dependent passes: a launch costs 1-2 us and every GMRES(3) sweep ends in a
// sum over the level.  Per-level launches took 65 us for one V-cycle from
// n = 127 down (gram 7.5, pre-smoothing 3, prolongation 3.7 us per level and
// sweep; one block for n <= 31: 9.5 + 3.5 + 9.5 us).
// One block per level set is bound by its SM's issue slots; clusters whose
// phases go through L2 paid ~4.7 us per phase.  Here the rows of every level
// are dealt to the blocks (R_k rows each, R_k = 2 R_{k+1}, so a block's
// coarse rows lie inside its fine rows), a block keeps its rows and four
// more on each side, forms the basis vectors redundantly on those, and only
// two kinds of phase cross blocks:
//   - the Gram sums (each block writes its ten sums to every peer, one
//     cluster barrier, every block solves the 3 x 3 system itself);
//   - the four halo rows of a new right-hand side, iterate or correction,
//     read from the owners' shared memory after a cluster barrier.
// A V-cycle over three levels and the coarsest solve takes 13 barriers.
//
// With `corr` > 0 the first level is the one of the ADR corrections: the
// launch runs `corr` corrections whole (residual and demodulation, V-cycle,
// modulation into the wave iterate, Algorithm 1), the iterate in shared
// memory throughout.
//
// The arithmetic per node is that of the per-level kernels
// (gmres_sstep.cuh, k_resdemod, the prolongation tile); sums are taken per
// thread, per warp, per block and over the blocks in rank order.  All threads
// of a cluster run the same phases, so every barrier is reached by all.
#pragma once
#include <cooperative_groups.h>

#include "gmres_sstep.cuh"

namespace wadr {

constexpr int CT_THREADS = 512, CT_WARPS = CT_THREADS / 32;
constexpr int CT_HALO = 4;      // rows kept on each side of a block's own
constexpr int CT_MAXL = 8;      // levels of a chain, the coarsest included

// Rows per block on level 0 of a chain of nl levels with ny rows: a multiple
// of 2^(nl-1), so that every level's share is twice the next one's.
__host__ __device__ constexpr int ct_rows(int ny, int nl, int cs) {
    const int d = 1 << (nl - 1);
    return (ny + cs * d - 1) / (cs * d) * d;
}
// the level's ADR coefficients are kept in shared memory (FP32) or read from
// L2 (FP64, whose vectors take the room)
template <typename T> __host__ __device__ constexpr bool ct_quads() { return sizeof(T) == 4; }
// Dynamic shared memory of a chain whose level 0 is n x ny: per level b and x
// (and the quads) on the block's rows and halo, three basis vectors of level
// 0, the coarsest right-hand side and, for whole corrections, the iterate.
template <typename T> __host__ __device__ constexpr long long ct_smem(int n, int ny, int nl, int cs, bool whole) {
    long long by = 16;   // the quads start on a 16-byte boundary
    int R = ct_rows(ny, nl, cs), nk = n, nyk = ny;
    const long long c = sizeof(cplx<T>);
    by += (3 + (whole ? 1 : 0)) * c * (R + 2 * CT_HALO) * (n + 2);
    for (int k = 0; k < nl; ++k) {
        by += (2 * c + (ct_quads<T>() ? (long long)sizeof(quad<T>) : 0)) * (R + 2 * CT_HALO) * (nk + 2);
        if (k == nl - 1) by += c * nk * nyk;
        R /= 2;
        nk /= 2;
        nyk /= 2;
    }
    return by;
}

// One level of a block's chain.
template <typename T> struct CtLevel {
    int n, ny, W, R, r0, r1;     // nodes per row, rows, row stride, rows per block, own rows [r0, r1)
    cplx<T> *B, *X;              // own and halo rows from row r0 - CT_HALO, one zero column on each side
    quad<T>* Q;
    T ih2, wh, s;
};

template <typename T, int CS>
__global__ void __launch_bounds__(CT_THREADS, 1) k_adr_cluster(const LevelDesc* __restrict__ D,
                                                               const int* __restrict__ chain, int corr) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char ct_smem_raw[];
    __shared__ LevelDesc Lv[CT_MAXL];
    __shared__ CtLevel<T> L[CT_MAXL];
    __shared__ int didx[CT_MAXL];
    __shared__ T shw[CT_WARPS * 16];
    __shared__ GsSum<T> part[2][CS][16];
    __shared__ T scl[S::NORM + 2];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid < CT_MAXL) didx[tid] = chain[(blockIdx.x / CS) * CT_MAXL + tid];
    __syncthreads();
    int nl = 0;
    while (nl < CT_MAXL && didx[nl] >= 0) ++nl;
    for (int k = w; k < nl; k += CT_WARPS) copy_desc(Lv[k], D + didx[k], lane);
    __syncthreads();
    cplx<T>* const K0 = reinterpret_cast<cplx<T>*>(ct_smem_raw);
    const int W0 = Lv[0].n + 2, R0 = ct_rows(Lv[0].ny, nl, CS), E0 = (R0 + 2 * CT_HALO) * W0;
    cplx<T>* const K1 = K0 + E0;
    cplx<T>* const K2 = K1 + E0;
    cplx<T>* const U = corr > 0 ? K2 + E0 : nullptr;
    cplx<T>* const Bd = K2 + (corr > 0 ? 2 : 1) * E0;           // dense coarsest right-hand side
    if (tid < nl) {
        unsigned char* p = reinterpret_cast<unsigned char*>(
            ((uintptr_t)(Bd + Lv[nl - 1].n * Lv[nl - 1].ny) + 15) & ~(uintptr_t)15);
        const size_t per = (ct_quads<T>() ? sizeof(quad<T>) : 0) + 2 * sizeof(cplx<T>);
        int R = R0;
        for (int k = 0; k < tid; ++k, R /= 2) p += (size_t)(R + 2 * CT_HALO) * (Lv[k].n + 2) * per;
        CtLevel<T>& l = L[tid];
        const LevelDesc& d = Lv[tid];
        l.n = d.n;
        l.ny = d.ny;
        l.W = d.n + 2;
        l.R = R;
        l.r0 = rank * R;
        l.r1 = min(l.r0 + R, d.ny);
        const int e = (R + 2 * CT_HALO) * l.W;
        l.Q = ct_quads<T>() ? reinterpret_cast<quad<T>*>(p) : nullptr;
        l.B = reinterpret_cast<cplx<T>*>(p + (ct_quads<T>() ? (size_t)e * sizeof(quad<T>) : 0));
        l.X = l.B + e;
        l.ih2 = LC<T>::ih2(d);
        l.wh = LC<T>::wh(d);
        l.s = LC<T>::gs(d);
    }
    __syncthreads();
    // f(local offset, row, column) for rows [r0 + a, r0 + R + b) of level l
    // that lie in the grid, columns in it; z(local offset) for the rows
    // outside and the two zero columns
    auto over = [&](const CtLevel<T>& l, int a, int b, auto&& f, auto&& z) {
        for (int q = a + w; q < l.R + b; q += CT_WARPS) {
            const int row = l.r0 + q, o = (q + CT_HALO) * l.W + 1;
            if ((unsigned)row < (unsigned)l.ny) {
                for (int c = lane; c < l.n; c += 32) f(o + c, row, c);
                if (lane < 2) z(o - 1 + lane * (l.n + 1));
            } else {
                for (int c = lane; c < l.W; c += 32) z(o - 1 + c);
            }
        }
    };
    auto none = [](int) {};
    // Constants of the setup and zeros first, so that this part may run beside
    // the end of the previous kernel: asynchronous copies of the quads of all
    // levels, then b, x and the iterate as zero (their halo columns and the
    // rows outside the grid are never written).
    if constexpr (ct_quads<T>())
        for (int k = 0; k + 1 < nl; ++k) {
            const quad<T>* const a = reinterpret_cast<const quad<T>*>(Lv[k].adr);
            const int pitch = Lv[k].pitch;
            quad<T>* const Q = L[k].Q;
            over(L[k], -3, 3,
                 [&](int o, int row, int c) { cp_async_elem(Q + o, a + (long long)row * pitch + c, true); }, none);
        }
    for (int k = 0; k < nl; ++k) {
        const int e = (L[k].R + 2 * CT_HALO) * L[k].W;
        for (int q = tid; q < 2 * e; q += CT_THREADS) L[k].B[q] = zero2<T>();
    }
    if (corr > 0)
        for (int q = tid; q < E0; q += CT_THREADS) U[q] = zero2<T>();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    cl.sync();   // every block of the cluster runs and its memory is set
    auto quad_at = [&](const CtLevel<T>& l, const LevelDesc& d, int o, int row, int c) {
        return ct_quads<T>() ? l.Q[o] : load_adr<T>(d, (long long)row * d.pitch + c);
    };
    // dst = s L src on rows [r0 + a, r0 + R + b)
    auto sl_rows = [&](const CtLevel<T>& l, const LevelDesc& d, const cplx<T>* src, cplx<T>* dst, int a, int b) {
        const T ih2 = l.ih2, wh = l.wh, s = l.s;
        const int W = l.W;
        over(l, a, b,
             [&](int o, int row, int c) {
                 dst[o] = cscale<T>(adr_pt<T>(quad_at(l, d, o, row, c), ih2, wh, src[o], src[o - 1], src[o + 1],
                                              src[o - W], src[o + W]), s);
             },
             [&](int o) { dst[o] = zero2<T>(); });
    };
    // rows [r0 - h, r0) and [r0 + R, r0 + R + h) of a level vector from their owners
    auto halo = [&](const CtLevel<T>& l, cplx<T>* v, int h) {
        for (int q = w; q < 2 * h; q += CT_WARPS) {
            const int row = q < h ? l.r0 - 1 - q : l.r0 + l.R + (q - h);
            if ((unsigned)row >= (unsigned)l.ny) continue;
            const int own = row / l.R;
            const cplx<T>* src = cl.map_shared_rank(v, own) + (row - own * l.R + CT_HALO) * l.W + 1;
            cplx<T>* dst = v + (row - l.r0 + CT_HALO) * l.W + 1;
            for (int c = lane; c < l.n; c += 32) dst[c] = src[c];
        }
    };
    // Gram sums of the cluster and the 3 x 3 solve (a cluster barrier inside);
    // the coefficients in scl of every block
    int par = 0;
    auto solve = [&](const GramAcc<T>& g) {
        cplx<T> ac[8];
        g.to_layout(ac);
        T v[16];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            v[2 * k] = ac[k].x;
            v[2 * k + 1] = ac[k].y;
        }
        const T ws = warp_sum16<T>(v, lane);
        if (!(lane & 1)) shw[w * 16 + (lane >> 1)] = ws;
        __syncthreads();
        if (w == 0) {
            const int id = lane >> 1, h = lane & 1;
            const GsSum<T> t = rows_sum16<T>(shw, CT_WARPS, lane);
#pragma unroll
            for (int p = 0; p < CS; p += 2) *cl.map_shared_rank(&part[par][rank][id], p + h) = t;
        }
        cl.sync();
        if (w == 0) gs_solve<T>(rows_sum16<T>(&part[par][0][0], CS, lane), lane, scl);
        par ^= 1;
        __syncthreads();
    };
    const LevelDesc& d0 = Lv[0];
    if (corr > 0) {
        const cplx<T>* u = slot<T>(d0, SU);
        over(L[0], -1, 1,
             [&](int o, int row, int c) { cp_async_elem(U + o, u + (long long)row * d0.pitch + c, true); }, none);
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
    }
    const int rounds = corr > 0 ? corr : 1;
    for (int m = 0; m < rounds; ++m) {
        if (corr > 0) {
            // b = exp(-i w phi) (g - A u) (k_resdemod) on the own rows
            const CtLevel<T>& l = L[0];
            const cplx<T>* g = slot<T>(d0, SG);
            const cplx<T>* mod = reinterpret_cast<const cplx<T>*>(d0.mod);
            const int W = l.W;
            over(l, 0, 0,
                 [&](int o, int row, int c) {
                     const long long p = (long long)row * d0.pitch + c;
                     const cplx<T> dg = helm_diag4<T>(d0, c, row, load_k<T>(d0, c, row), load_sig<T>(d0, c, row));
                     const cplx<T> r = csub<T>(__ldg(g + p), helm_diff<T>(dg, U[o], U[o - 1], U[o + 1], U[o - W],
                                                                          U[o + W], l.ih2));
                     l.B[o] = cmulc<T>(__ldg(mod + p), r);
                 },
                 none);
            cl.sync();
            halo(l, l.B, CT_HALO);
        } else {
            const cplx<T>* b = slot<T>(d0, SAB);
            cplx<T>* const B0 = L[0].B;
            over(L[0], -CT_HALO, CT_HALO,
                 [&](int o, int row, int c) { cp_async_elem(B0 + o, b + (long long)row * d0.pitch + c, true); }, none);
            cp_async_commit();
            cp_async_wait<0>();
        }
        __syncthreads();
        // the first 256 values of a row of the inverse; this warp's first row
        // (FP32) is fetched while the last level above the coarsest is smoothed
        const int N = L[nl - 1].n * L[nl - 1].ny, p0 = L[nl - 1].r0 * L[nl - 1].n + w, p1 = L[nl - 1].r1 * L[nl - 1].n;
        const cplx<T>* const inv = reinterpret_cast<const cplx<T>*>(Lv[nl - 1].inv_adr);
        constexpr bool early = ct_quads<T>();   // (FP64 has no registers to spare)
        cplx<T> av[8];
        auto fetch = [&](int p) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int q = lane + 32 * u;
                av[u] = q < N ? __ldg(inv + (long long)p * N + q) : zero2<T>();
            }
        };
        // down: GMRES(3) from x = 0, x kept, the residual restricted to the next b
        for (int k = 0; k + 1 < nl; ++k) {
            const CtLevel<T>& l = L[k];
            const LevelDesc& d = Lv[k];
            sl_rows(l, d, l.B, K1, -3, 3);
            __syncthreads();
            sl_rows(l, d, K1, K2, -2, 2);
            __syncthreads();
            GramAcc<T> g;
            g.zero();
            const int W = l.W;
            {
                const T ih2 = l.ih2, wh = l.wh, s = l.s;
                over(l, -1, 1,
                     [&](int o, int row, int c) {
                         const cplx<T> k3 = cscale<T>(adr_pt<T>(quad_at(l, d, o, row, c), ih2, wh, K2[o], K2[o - 1],
                                                                K2[o + 1], K2[o - W], K2[o + W]), s);
                         K0[o] = k3;
                         if (row >= l.r0 && row < l.r1) gram_acc<T>(g, l.B[o], K1[o], K2[o], k3);
                     },
                     [&](int o) { K0[o] = zero2<T>(); });
            }
            solve(g);
            if (early && k + 2 == nl && p0 < p1) fetch(p0);
            {
                const cplx<T> c0 = sload2<T>(scl, S::GC), c1 = sload2<T>(scl, S::GC + 2), c2 = sload2<T>(scl, S::GC + 4);
                const cplx<T> sc0 = cscale<T>(c0, l.s), sc1 = cscale<T>(c1, l.s), sc2 = cscale<T>(c2, l.s);
                over(l, -1, 1,
                     [&](int o, int row, int) {
                         const cplx<T> k0 = l.B[o], k1 = K1[o], k2 = K2[o];
                         if (row >= l.r0 && row < l.r1)
                             l.X[o] = cfma<T>(sc2, k2, cfma<T>(sc1, k1, cmul<T>(sc0, k0)));
                         cplx<T> v = csub<T>(k0, cmul<T>(c0, k1));
                         v = csub<T>(v, cmul<T>(c1, k2));
                         K0[o] = csub<T>(v, cmul<T>(c2, K0[o]));
                     },
                     none);
            }
            __syncthreads();
            {
                // full weighting; coarse node (I, J) on fine node (2I+1, 2J+1)
                const CtLevel<T>& lc = L[k + 1];
                const int r0 = l.r0;
                over(lc, 0, 0,
                     [&](int o, int J, int I) {
                         const cplx<T>* q = K0 + (2 * J + 1 - r0 + CT_HALO) * W + 2 * I + 2;
                         const cplx<T> s2 = cadd<T>(cadd<T>(q[-1], q[1]), cadd<T>(q[-W], q[W]));
                         const cplx<T> s1 = cadd<T>(cadd<T>(q[-W - 1], q[-W + 1]), cadd<T>(q[W - 1], q[W + 1]));
                         lc.B[o] = cscale<T>(cadd<T>(cadd<T>(cscale<T>(q[0], T(4)), cscale<T>(s2, T(2))), s1), T(0.0625));
                     },
                     none);
            }
            cl.sync();
            if (k + 2 < nl) halo(L[k + 1], L[k + 1].B, CT_HALO);
            halo(l, l.X, CT_HALO);
            __syncthreads();
        }
        {
            // coarsest solve: the whole right-hand side in every block, a warp per own row of the inverse
            const CtLevel<T>& l = L[nl - 1];
            const int n = l.n;
            for (int row = w; row < l.ny; row += CT_WARPS) {
                const int own = row / l.R;
                const cplx<T>* src = cl.map_shared_rank(l.B, own) + (row - own * l.R + CT_HALO) * l.W + 1;
                for (int c = lane; c < n; c += 32) Bd[row * n + c] = src[c];
            }
            __syncthreads();
            for (int p = p0; p < p1; p += CT_WARPS) {
                if (!early || p != p0 || nl < 2) fetch(p);
                // as k_coarse: four independent accumulators
                cplx<T> ac[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) ac[u] = zero2<T>();
                auto add = [&](int u, int q, cplx<T> a) {
                    if (q < N) {
                        const cplx<T> bv = Bd[q];
                        ac[u].x = fma(a.x, bv.x, ac[u].x);
                        ac[u].x = fma(-a.y, bv.y, ac[u].x);
                        ac[u].y = fma(a.x, bv.y, ac[u].y);
                        ac[u].y = fma(a.y, bv.x, ac[u].y);
                    }
                };
#pragma unroll
                for (int u = 0; u < 8; ++u) add(u & 3, lane + 32 * u, av[u]);
                for (int q0 = lane + 256; q0 < N; q0 += 128)
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int q = q0 + 32 * u;
                        add(u, q, q < N ? __ldg(inv + (long long)p * N + q) : zero2<T>());
                    }
                cplx<T> acc = cadd<T>(cadd<T>(ac[0], ac[1]), cadd<T>(ac[2], ac[3]));
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    acc.x += __shfl_down_sync(0xffffffffu, acc.x, o);
                    acc.y += __shfl_down_sync(0xffffffffu, acc.y, o);
                }
                if (lane == 0) {
                    const int row = p / n;
                    l.X[(row - l.r0 + CT_HALO) * l.W + 1 + p - row * n] = acc;
                }
            }
            cl.sync();
        }
        // up: x' = x + P e, r0 = b - L x', GMRES(3) from x'
        for (int k = nl - 2; k >= 0; --k) {
            const CtLevel<T>& l = L[k];
            const CtLevel<T>& lc = L[k + 1];
            const LevelDesc& d = Lv[k];
            const int W = l.W, Wc = lc.W;
            halo(lc, lc.X, CT_HALO);
            __syncthreads();
            over(l, -CT_HALO, CT_HALO,
                 [&](int o, int row, int c) {
                     // bilinear: (1, 0) for odd nodes, (1/2, 1/2) for even ones
                     const int ia = (c - 1) >> 1, ja = (row - 1) >> 1;
                     const T wa0 = (c & 1) ? T(1) : T(0.5), wa1 = T(1) - wa0;
                     const T wb0 = (row & 1) ? T(1) : T(0.5), wb1 = T(1) - wb0;
                     const cplx<T>* e = lc.X + (ja - lc.r0 + CT_HALO) * Wc + ia + 1;
                     cplx<T> v = cscale<T>(cadd<T>(cscale<T>(e[0], wa0), cscale<T>(e[1], wa1)), wb0);
                     v = cadd<T>(v, cscale<T>(cadd<T>(cscale<T>(e[Wc], wa0), cscale<T>(e[Wc + 1], wa1)), wb1));
                     l.X[o] = cadd<T>(l.X[o], v);
                 },
                 none);
            __syncthreads();
            const T ih2 = l.ih2, wh = l.wh, s = l.s;
            over(l, -3, 3,
                 [&](int o, int row, int c) {
                     const cplx<T>* x = l.X + o;
                     K0[o] = csub<T>(l.B[o], adr_pt<T>(quad_at(l, d, o, row, c), ih2, wh, x[0], x[-1], x[1], x[-W], x[W]));
                 },
                 [&](int o) { K0[o] = zero2<T>(); });
            __syncthreads();
            sl_rows(l, d, K0, K1, -2, 2);
            __syncthreads();
            sl_rows(l, d, K1, K2, -1, 1);
            __syncthreads();
            GramAcc<T> g;
            g.zero();
            over(l, 0, 0,
                 [&](int o, int row, int c) {
                     const cplx<T> k3 = cscale<T>(adr_pt<T>(quad_at(l, d, o, row, c), ih2, wh, K2[o], K2[o - 1],
                                                            K2[o + 1], K2[o - W], K2[o + W]), s);
                     gram_acc<T>(g, K0[o], K1[o], K2[o], k3);
                 },
                 none);
            solve(g);
            const cplx<T> c0 = cscale<T>(sload2<T>(scl, S::GC), s), c1 = cscale<T>(sload2<T>(scl, S::GC + 2), s),
                          c2 = cscale<T>(sload2<T>(scl, S::GC + 4), s);
            const cplx<T>* mod = reinterpret_cast<const cplx<T>*>(d0.mod);
            over(l, 0, 0,
                 [&](int o, int row, int c) {
                     const cplx<T> x = cfma<T>(c2, K2[o], cfma<T>(c1, K1[o], cfma<T>(c0, K0[o], l.X[o])));
                     if (k > 0) l.X[o] = x;
                     else if (corr > 0) U[o] = cfma<T>(__ldg(mod + (long long)row * d0.pitch + c), x, U[o]);
                     else slot<T>(d0, SAX)[(long long)row * d0.pitch + c] = x;
                 },
                 none);
            cl.sync();   // (after the last level: no block leaves while a peer may still read its rows)
        }
        if (corr > 0) {
            halo(L[0], U, 1);
            __syncthreads();
        }
    }
    if (corr > 0) {
        cplx<T>* u = slot<T>(d0, SU);
        over(L[0], 0, 0, [&](int o, int row, int c) { u[(long long)row * d0.pitch + c] = U[o]; }, none);
        cl.sync();
    }
}

}  // namespace wadr
