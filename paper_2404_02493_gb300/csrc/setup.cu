// Setup kernels (FP64): coefficient injection, ADR coefficients, level-2
// modulation, the Gershgorin bound of A^*A and the coarsest-level inverses.
// These run once per mg_setup; none is on the per-cycle path.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "handle.h"
#include "setup_kernels.cuh"

namespace wadr {

// Coefficients of level `level` by injection from the fine grid: coarse node
// I of level l sits on fine node 2^(l-1) (I+1) - 1 (Algorithm 1's
// re-discretised operator A_H; coefficients sampled at coinciding nodes).
__global__ void k_inject(const double* __restrict__ kf, const double* __restrict__ pf, int n1, int ny1,
                         double omega, int bc, double swidth, double spower, int level, double* k64, double* phi64,
                         double* sig64, int n, int ny, int pitch) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= n || j >= ny) return;
    const long long f = 1LL << (level - 1);
    const long long fi = f * (i + 1) - 1, fj = f * (j + 1) - 1;
    const long long q = fj * n1 + fi, p = (long long)j * pitch + i;
    const double k = kf[q];
    k64[p] = k;
    phi64[p] = pf[q];
    if (sig64) {
        // sponge mask: gamma(d) = omega ((W-d)/W)^p for d < W = width 2 pi/omega
        // (default one wavelength, p = 2),
        // d = distance of the fine node to the boundary of [0, lx] x [0, ly]
        // (the longer side has unit length, h1 = 1/(max(n1, ny1)+1));
        // sig = omega gamma s^2
        const int m1 = max(n1, ny1);
        const double h1 = 1.0 / (m1 + 1);
        const double lx = n1 == m1 ? 1.0 : (n1 + 1) * h1, ly = ny1 == m1 ? 1.0 : (ny1 + 1) * h1;
        const double x = (fi + 1) * h1, y = (fj + 1) * h1;
        const double dist = fmin(fmin(x, lx - x), fmin(y, ly - y));
        const double W = swidth == 1.0 ? 2.0 * M_PI / omega : swidth * (2.0 * M_PI / omega);
        const double t = (W - dist) / W;
        const double gam = dist < W ? (spower == 2.0 ? omega * t * t : omega * pow(t, spower)) : 0.0;
        sig64[p] = omega * gam * (k / omega) * (k / omega);
    }
}

void setup_inject(const double* k_fine, const double* phi_fine, int n1, int ny1, double omega, int bc,
                  double sponge_width, double sponge_power, int level, double* k64, double* phi64, double* sig64, int n,
                  int ny, int pitch, cudaStream_t st) {
    dim3 b(32, 8), g((n + 31) / 32, (ny + 7) / 8);
    k_inject<<<g, b, 0, st>>>(k_fine, phi_fine, n1, ny1, omega, bc, sponge_width, sponge_power, level, k64, phi64,
                              sig64, n, ny, pitch);
}

// Wave-Ray plane-wave phase cx x + cy y on level l (scale = 2^(l-1), h1 the
// level-1 spacing), as injection of the level-1 phase places it
void setup_plane_phase(double* phi64, int n, int ny, int pitch, double h1, int scale, double cx, double cy,
                       cudaStream_t st) {
    dim3 b(32, 8), g((n + 31) / 32, (ny + 7) / 8);
    k_plane_phase<<<g, b, 0, st>>>(phi64, n, ny, pitch, h1, scale, cx, cy);
}

// Input validation of one instance's fine fields (dense n x ny): counts the
// nodes whose k is not a finite positive number (out[0]) and whose phi is
// not finite (out[1]).
__global__ void k_check_fields(const double* __restrict__ k, const double* __restrict__ phi, long long npt,
                               unsigned long long* out) {
    unsigned long long bad_k = 0, bad_phi = 0;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < npt; p += (long long)gridDim.x * blockDim.x) {
        const double kv = k[p], pv = phi[p];
        bad_k += !(isfinite(kv) && kv > 0.0);
        bad_phi += !isfinite(pv);
    }
    if (bad_k) atomicAdd(out, bad_k);
    if (bad_phi) atomicAdd(out + 1, bad_phi);
}

int setup_check_fields(const double* k, const double* phi, int n, int ny, double* dscratch, long long* bad_k,
                       long long* bad_phi, cudaStream_t st) {
    unsigned long long* o = reinterpret_cast<unsigned long long*>(dscratch);
    WADR_CHECK(cudaMemsetAsync(o, 0, 2 * sizeof(unsigned long long), st));
    const long long npt = (long long)n * ny;
    const int blocks = (int)std::min<long long>((npt + 255) / 256, 1216);
    k_check_fields<<<blocks, 256, 0, st>>>(k, phi, npt, o);
    WADR_CHECK(cudaGetLastError());
    unsigned long long v[2] = {0, 0};
    WADR_CHECK(cudaMemcpyAsync(v, o, sizeof(v), cudaMemcpyDeviceToHost, st));
    WADR_CHECK(cudaStreamSynchronize(st));
    *bad_k = (long long)v[0];
    *bad_phi = (long long)v[1];
    return MG_OK;
}

// Peclet number of an ADR level (Section 3.2.2: the central-difference ADR
// discretisation needs 2 omega h max(|phi_x|, |phi_y|) <= 2): the maximum over
// nodes of omega h max(|phi_x|, |phi_y|), with the same phase derivatives as
// the ADR coefficients.  The condition holds where the value is <= 1.
__global__ void k_peclet(const double* phi64, const double* k64, const double* sig64, int n, int ny, int pitch,
                         double h, double omega, int bc, unsigned long long* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= n || j >= ny) return;
    const AdrCoef c = adr_coef_at(phi64, k64, sig64, n, ny, pitch, h, omega, bc, 0.0, i, j, 0);
    const double v = omega * h * fmax(fabs(c.px), fabs(c.py));
    atomicMax(out, (unsigned long long)__double_as_longlong(v));
}

double setup_peclet(const double* k64, const double* phi64, const double* sig64, int n, int ny, int pitch, double h,
                    double omega, int bc, double* dscratch, cudaStream_t st) {
    unsigned long long* o = reinterpret_cast<unsigned long long*>(dscratch);
    cudaMemsetAsync(o, 0, sizeof(unsigned long long), st);
    dim3 b(32, 8), g((n + 31) / 32, (ny + 7) / 8);
    k_peclet<<<g, b, 0, st>>>(phi64, k64, sig64, n, ny, pitch, h, omega, bc, o);
    unsigned long long v = 0;
    cudaMemcpyAsync(&v, o, sizeof(v), cudaMemcpyDeviceToHost, st);
    cudaStreamSynchronize(st);
    double r;
    memcpy(&r, &v, sizeof(r));
    return r;
}

// max over nodes of the absolute row sum |A_pp| + (in-grid neighbours)/h^2
__device__ __forceinline__ double helm_row_sum(const double* k64, const double* sig64, int n, int ny, int pitch,
                                               double h, int bc, double shift, int i, int j) {
    const long long p = (long long)j * pitch + i;
    const double k = k64[p], kh = k * h;
    double re = 4.0 - kh * kh, im = 0.0;
    const int m = (i == 0) + (i == n - 1) + (j == 0) + (j == ny - 1);
    if (bc == BC_ABC1) {
        re -= m;
        im -= m * kh;
    } else if (bc == BC_SPONGE) {
        im -= h * h * sig64[p];
    }
    if (shift != 0.0) im -= shift * kh * kh;
    return (sqrt(re * re + im * im) + (4 - m)) / (h * h);
}

__global__ void k_gersh(const double* k64, const double* sig64, int n, int ny, int pitch, double h, int bc,
                        double shift, unsigned long long* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= n || j >= ny) return;
    const double v = helm_row_sum(k64, sig64, n, ny, pitch, h, bc, shift, i, j);
    // positive doubles order like their bit patterns
    atomicMax(out, (unsigned long long)__double_as_longlong(v));
}

double setup_lambda_max(const double* k64, const double* sig64, int n, int ny, int pitch, double h, int bc,
                        double shift, double* dscratch, cudaStream_t st) {
    unsigned long long* o = reinterpret_cast<unsigned long long*>(dscratch);
    cudaMemsetAsync(o, 0, sizeof(unsigned long long), st);
    dim3 b(32, 8), g((n + 31) / 32, (ny + 7) / 8);
    k_gersh<<<g, b, 0, st>>>(k64, sig64, n, ny, pitch, h, bc, shift, o);
    unsigned long long v = 0;
    cudaMemcpyAsync(&v, o, sizeof(v), cudaMemcpyDeviceToHost, st);
    cudaStreamSynchronize(st);
    double r;
    memcpy(&r, &v, sizeof(r));
    return r * r;
}

// max over nodes of the absolute row sum of the ADR operator |d| + sum |c_dir|
__global__ void k_adr_rowmax(const double* phi64, const double* k64, const double* sig64, int n, int ny, int pitch,
                             double h, double omega, int bc, double shift, int adr_flags, unsigned long long* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= n || j >= ny) return;
    const AdrCoef c = adr_coef_at(phi64, k64, sig64, n, ny, pitch, h, omega, bc, shift, i, j, adr_flags);
    const double v = sqrt(dabs2(c.d)) + sqrt(dabs2(c.cw)) + sqrt(dabs2(c.ce)) + sqrt(dabs2(c.cs)) +
                     sqrt(dabs2(c.cn));
    atomicMax(out, (unsigned long long)__double_as_longlong(v));
}

// Scale of the s-step GMRES basis of an ADR level: the power of two s with
// s * (max row sum of |L|) in (1/2, 1], so that ||s L||_inf <= 1 and the
// basis vectors (s L)^j r0 stay O(|r0|) without rounding from s itself.
double setup_adr_scale(const double* k64, const double* phi64, const double* sig64, int n, int ny, int pitch,
                       double h, double omega, int bc, double shift, int adr_flags, double* dscratch,
                       cudaStream_t st) {
    unsigned long long* o = reinterpret_cast<unsigned long long*>(dscratch);
    cudaMemsetAsync(o, 0, sizeof(unsigned long long), st);
    dim3 b(32, 8), g((n + 31) / 32, (ny + 7) / 8);
    k_adr_rowmax<<<g, b, 0, st>>>(phi64, k64, sig64, n, ny, pitch, h, omega, bc, shift, adr_flags, o);
    unsigned long long v = 0;
    cudaMemcpyAsync(&v, o, sizeof(v), cudaMemcpyDeviceToHost, st);
    cudaStreamSynchronize(st);
    double r;
    memcpy(&r, &v, sizeof(r));
    if (!(r > 0.0)) return 1.0;
    int e;
    std::frexp(r, &e);          // r = f 2^e, f in [1/2, 1)
    return std::ldexp(1.0, -e);
}

// ---------------------------------------------------------------- coarsest-level inverses
// Dense inverses of the coarsest operators (N = n ny <= 1024, row p = j*n + i)
// in FP64: Gauss-Jordan elimination in place with partial pivoting, blocked
// over panels of GJB columns, all matrices of a setup together (both operators
// of every instance; one grid slice per matrix).  Per panel two launches:
//   k_gj_panel   one block per matrix eliminates the panel's columns in
//                shared memory: pivot of column k = largest modulus among the
//                rows >= k (smallest index on ties); leaves P = D in the pivot
//                rows K and -A_RK D elsewhere (D = A_KK^-1) and the row swaps
//   k_gj_update  the remaining columns, out of place (the old pivot rows are
//                read by every block): A'_ic (i not in K) + sum_j P_ij A'_{K_j c}
// What bounds it: N complex multiply-adds per entry (N^3 in all) on the FP64
// pipes of 2 lanes per SM and clock, and a chain of N pivot steps.  One block
// doing the whole factorisation (and one thread per column the triangular
// solves) held a single SM's pipe and took 7.5 + 12.1 ms per 225 x 225 matrix;
// the panels keep only N^2 GJB of the work in one block and the rest runs on
// all SMs (figures at setup_coarse_inverses).
constexpr int GJB = 8;               // panel columns: N x 8 complex FP64 (128 KB at N = 1024) fit a block
constexpr int GJT = 512;             // panel threads
constexpr int GJX = 32, GJY = 16;    // update tile (columns x rows), 256 threads

struct GjMat {
    CoarseJob c;
    int N;
    double2 *A, *B;                  // ping-pong matrices
    double2* P;                      // panel, N x GJB row-major
    int *src, *perm, *info;          // this panel's row sources, row order so far, singular flag
};

// the five entries of row p (the matrix is zeroed before)
__global__ void k_gj_dense(const GjMat* __restrict__ M) {
    const GjMat& m = M[blockIdx.y];
    const CoarseJob& c = m.c;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int N = m.N, n = c.n, ny = c.ny;
    if (p >= N) return;
    m.perm[p] = p;
    if (p == 0) *m.info = 0;
    const int i = p % n, j = p / n;
    double2* row = m.A + (long long)p * N;
    const double ih2 = 1.0 / (c.h * c.h);
    if (c.which == 0) {
        const long long pp = (long long)j * c.pitch + i;
        const double k = c.k64[pp], kh = k * c.h;
        double re = 4.0 - kh * kh, im = 0.0;
        const int miss = (i == 0) + (i == n - 1) + (j == 0) + (j == ny - 1);
        if (c.bc == BC_ABC1) { re -= miss; im -= miss * kh; }
        else if (c.bc == BC_SPONGE) { im -= c.h * c.h * c.sig64[pp]; }
        if (c.shift != 0.0) im -= c.shift * kh * kh;
        row[p] = make_double2(re * ih2, im * ih2);
        if (i > 0) row[p - 1] = make_double2(-ih2, 0);
        if (i < n - 1) row[p + 1] = make_double2(-ih2, 0);
        if (j > 0) row[p - n] = make_double2(-ih2, 0);
        if (j < ny - 1) row[p + n] = make_double2(-ih2, 0);
    } else {
        const AdrCoef a = adr_coef_at(c.phi64, c.k64, c.sig64, n, ny, c.pitch, c.h, c.omega, c.bc, c.shift, i, j,
                                      c.adr_flags);
        row[p] = a.d;
        if (i > 0) row[p - 1] = a.cw;
        if (i < n - 1) row[p + 1] = a.ce;
        if (j > 0) row[p - n] = a.cs;
        if (j < ny - 1) row[p + n] = a.cn;
    }
}

// Panel of columns [k0, k0 + GJB): thread t holds rows t, t + GJT of the
// panel's shared-memory columns (column-major, so a warp's rows are
// contiguous).  The divisions of a pivot run in one warp: a warp's FP64
// instruction holds the pipe for 16 cycles, so redundant copies would queue.
__global__ void __launch_bounds__(GJT) k_gj_panel(const GjMat* __restrict__ M, int step) {
    extern __shared__ __align__(16) unsigned char gj_smem[];
    __shared__ unsigned long long wkey[GJT / 32];
    __shared__ int wrow[GJT / 32];
    __shared__ double2 rk[GJB];
    const GjMat& m = M[blockIdx.x];
    const int N = m.N, k0 = step * GJB;
    if (k0 >= N) return;
    const int b = min(GJB, N - k0);
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    double2* const Pc = reinterpret_cast<double2*>(gj_smem);     // [GJB][N]
    int* const src = reinterpret_cast<int*>(Pc + (size_t)GJB * N);
    const double2* A = (step & 1) ? m.B : m.A;
    for (int e = t; e < N * GJB; e += GJT) {
        const int i = e / GJB, c = e % GJB;
        if (c < b) Pc[(size_t)c * N + i] = A[(long long)i * N + k0 + c];
    }
    for (int i = t; i < N; i += GJT) src[i] = i;
    __syncthreads();
    for (int j = 0; j < b; ++j) {
        const int k = k0 + j;
        double2* const col = Pc + (size_t)j * N;
        // largest modulus, smallest row on ties (positive doubles order like
        // their bit patterns; NaN counts as zero)
        unsigned long long key = 0;
        int row = k;
        for (int i = k + t; i < N; i += GJT) {
            const double v = dabs2(col[i]);
            const unsigned long long q = v > 0.0 ? (unsigned long long)__double_as_longlong(v) : 0ull;
            if (q > key) { key = q; row = i; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long q = __shfl_xor_sync(0xffffffffu, key, o);
            const int r = __shfl_xor_sync(0xffffffffu, row, o);
            if (q > key || (q == key && r < row)) { key = q; row = r; }
        }
        if (lane == 0) { wkey[w] = key; wrow[w] = row; }
        __syncthreads();
        if (w == 0) {
            key = lane < GJT / 32 ? wkey[lane] : 0ull;
            row = lane < GJT / 32 ? wrow[lane] : N;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long q = __shfl_xor_sync(0xffffffffu, key, o);
                const int r = __shfl_xor_sync(0xffffffffu, row, o);
                if (q > key || (q == key && r < row)) { key = q; row = r; }
            }
            const int p = key ? row : k;
            if (lane < b) {
                // scaled pivot row; the row it replaces moves to row p
                const double2 piv = col[p];
                const double2 pinv = key ? ddiv(make_double2(1.0, 0.0), piv) : make_double2(0.0, 0.0);
                const double2 v = Pc[(size_t)lane * N + p], old = Pc[(size_t)lane * N + k];
                __syncwarp((1u << b) - 1u);
                const double2 r = lane == j ? pinv : dmul(v, pinv);
                rk[lane] = r;
                Pc[(size_t)lane * N + p] = old;
                Pc[(size_t)lane * N + k] = r;
            }
            if (lane == 0) {
                if (!key) *m.info = k + 1;
                const int s = src[k];
                src[k] = src[p];
                src[p] = s;
                const int q = m.perm[k];
                m.perm[k] = m.perm[p];
                m.perm[p] = q;
            }
        }
        __syncthreads();
        for (int i = t; i < N; i += GJT) {
            if (i == k) continue;
            const double2 f = col[i];
#pragma unroll
            for (int c = 0; c < GJB; ++c) {
                if (c >= b) break;
                if (c != j) Pc[(size_t)c * N + i] = dsub(Pc[(size_t)c * N + i], dmul(f, rk[c]));
            }
            const double2 g = dmul(f, rk[j]);
            col[i] = make_double2(-g.x, -g.y);
        }
        __syncthreads();
    }
    for (int e = t; e < N * GJB; e += GJT) {
        const int i = e / GJB, c = e % GJB;
        if (c < b) m.P[e] = Pc[(size_t)c * N + i];
    }
    for (int i = t; i < N; i += GJT) m.src[i] = src[i];
}

__global__ void __launch_bounds__(256) k_gj_update(const GjMat* __restrict__ M, int step) {
    __shared__ double2 Ps[GJY][GJB];
    __shared__ double2 As[GJB][GJX];
    const GjMat& m = M[blockIdx.y];
    const int N = m.N, k0 = step * GJB;
    if (k0 >= N) return;
    const int b = min(GJB, N - k0);
    const int ntx = (N + GJX - 1) / GJX;
    const int c0 = (blockIdx.x % ntx) * GJX, i0 = (blockIdx.x / ntx) * GJY;
    if (i0 >= N) return;
    const double2* A = (step & 1) ? m.B : m.A;
    double2* O = (step & 1) ? m.A : m.B;
    const int t = threadIdx.x;
    if (t < GJY * GJB) {
        const int r = t / GJB, j = t % GJB;
        Ps[r][j] = (i0 + r < N && j < b) ? m.P[(i0 + r) * GJB + j] : make_double2(0.0, 0.0);
    }
    {
        const int j = t / GJX, c = t % GJX;
        As[j][c] = (j < b && c0 + c < N) ? A[(long long)m.src[k0 + j] * N + c0 + c] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    const int c = t % GJX, gc = c0 + c;
#pragma unroll
    for (int q = 0; q < GJY / 8; ++q) {
        const int r = t / GJX + 8 * q, i = i0 + r;
        if (i >= N || gc >= N) continue;
        double2 v;
        if (gc >= k0 && gc < k0 + b) {
            v = Ps[r][gc - k0];
        } else {
            v = (i >= k0 && i < k0 + b) ? make_double2(0.0, 0.0) : A[(long long)m.src[i] * N + gc];
#pragma unroll
            for (int j = 0; j < GJB; ++j) {
                const double2 p = Ps[r][j], a = As[j][c];
                v.x = fma(p.x, a.x, v.x);
                v.y = fma(p.x, a.y, v.y);
                v.x = fma(-p.y, a.y, v.x);
                v.y = fma(p.y, a.x, v.y);
            }
        }
        O[(long long)i * N + gc] = v;
    }
}

// column c of the eliminated matrix is column perm[c] of the inverse; stored
// in the cycle precision (single: rounded to complex FP32)
__global__ void k_gj_store(const GjMat* __restrict__ M) {
    const GjMat& m = M[blockIdx.y];
    const int N = m.N, steps = (N + GJB - 1) / GJB;
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)N * N) return;
    const int i = (int)(e / N), c = (int)(e % N);
    const double2 v = ((steps & 1) ? m.B : m.A)[e];
    const long long o = (long long)i * N + m.perm[c];
    if (m.c.single) reinterpret_cast<float2*>(m.c.inv)[o] = make_float2((float)v.x, (float)v.y);
    else reinterpret_cast<double2*>(m.c.inv)[o] = v;
}

// The inverses of all jobs (always eliminated in FP64; see CoarseJob).  The
// temporary matrices of one group of jobs stay below 256 MB (or one job), and
// where the memory for a group is not there, below half of what was asked.
// Two 225 x 225 inverses: 39.2 ms one block per matrix -> 1.8 ms (29 panels of 49 us, 29 updates of 13 us).
int setup_coarse_inverses(const std::vector<CoarseJob>& jobs, cudaStream_t st) {
    static_assert(GJX * GJB == 256 && GJX * 8 == 256 && GJY * GJB <= 256, "update tile");
    size_t group = 256u << 20, q0 = 0;
    while (q0 < jobs.size()) {
        size_t q1 = q0, bytes = 0;
        int nmax = 0;
        std::vector<size_t> at;
        while (q1 < jobs.size()) {
            const size_t N = (size_t)jobs[q1].n * jobs[q1].ny;
            const size_t need = (2 * N * N + N * GJB) * sizeof(double2) + (2 * N * sizeof(int) + 255) / 256 * 256;
            if (q1 > q0 && (bytes + need > group || q1 - q0 >= 32768)) break;   // (a grid slice per job)
            at.push_back(bytes);
            bytes += need;
            nmax = std::max(nmax, (int)N);
            ++q1;
        }
        const size_t nj = q1 - q0, infos = (nj * sizeof(GjMat) + 255) / 256 * 256,
                     mats = infos + (nj * sizeof(int) + 255) / 256 * 256;
        unsigned char* base = nullptr;
        if (cudaMalloc(&base, mats + bytes) != cudaSuccess) {
            cudaGetLastError();
            if (nj > 1) {
                group = bytes / 2;
                continue;
            }
            set_error("mg_setup: out of device memory (coarsest-level inverse)");
            return MG_ENOMEM;
        }
        std::vector<GjMat> hm(nj);
        std::vector<int> info(nj, 0);
        for (size_t q = 0; q < nj; ++q) {
            GjMat& m = hm[q];
            m.c = jobs[q0 + q];
            m.N = m.c.n * m.c.ny;
            const size_t N = (size_t)m.N;
            m.A = (double2*)(base + mats + at[q]);
            m.B = m.A + N * N;
            m.P = m.B + N * N;
            m.src = (int*)(m.P + N * GJB);
            m.perm = m.src + N;
            m.info = (int*)(base + infos) + q;
        }
        const GjMat* dm = (const GjMat*)base;
        auto run = [&]() -> cudaError_t {
            cudaError_t e = cudaMemcpyAsync(base, hm.data(), nj * sizeof(GjMat), cudaMemcpyHostToDevice, st);
            if (e != cudaSuccess) return e;
            if ((e = cudaMemsetAsync(base + mats, 0, bytes, st)) != cudaSuccess) return e;
            const int smem = nmax * GJB * (int)sizeof(double2) + nmax * (int)sizeof(int);
            if ((e = cudaFuncSetAttribute(k_gj_panel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          MAX_COARSE_NODES * (GJB * (int)sizeof(double2) + (int)sizeof(int)))) !=
                cudaSuccess)
                return e;
            const unsigned ntile = (unsigned)((nmax + GJX - 1) / GJX) * (unsigned)((nmax + GJY - 1) / GJY);
            k_gj_dense<<<dim3((nmax + 127) / 128, (unsigned)nj), 128, 0, st>>>(dm);
            for (int s = 0; s * GJB < nmax; ++s) {
                k_gj_panel<<<(unsigned)nj, GJT, smem, st>>>(dm, s);
                k_gj_update<<<dim3(ntile, (unsigned)nj), 256, 0, st>>>(dm, s);
            }
            k_gj_store<<<dim3((unsigned)(((size_t)nmax * nmax + 255) / 256), (unsigned)nj), 256, 0, st>>>(dm);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            return cudaMemcpyAsync(info.data(), base + infos, nj * sizeof(int), cudaMemcpyDeviceToHost, st);
        };
        cudaError_t e = run();
        const cudaError_t es = cudaStreamSynchronize(st);
        if (e == cudaSuccess) e = es;
        cudaFree(base);
        if (e != cudaSuccess) {
            set_error(std::string("coarse inverse: ") + cudaGetErrorString(e));
            return MG_ECUDA;
        }
        for (int v : info)
            if (v != 0) {
                set_error("coarse inverse: singular coarsest operator");
                return MG_EINVAL;
            }
        q0 = q1;
    }
    return MG_OK;
}

}  // namespace wadr
