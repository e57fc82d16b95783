// Travel-time phase on the device: the first-order Godunov discretisation of
// the eikonal equation |grad tau| = s, tau(x0) = 0 (Section 3.2, eq.
// eikeq), the phase the ADR correction takes as input (Section 3.2.1 obtains
// it from a network trained on eikonal solutions; here it is computed).
//
// Discrete problem: at every node not fixed by the source,
//   a = min(tau_W, tau_E), b = min(tau_S, tau_N), f = s h,
//   tau = min(a, b) + f                          if |a - b| >= f,
//   tau = (a + b + sqrt(2 f^2 - (a - b)^2)) / 2  otherwise,
// and nodes within r_init of x0 hold s(x0) |x - x0| (s at the node nearest
// x0).  The update is monotone: from tau = inf every order of updates
// decreases the values to the same fixed point (Zhao's fast sweeping does it
// by Gauss-Seidel sweeps in four orderings over the whole grid).
//
// GB300 layout: the grid is cut into 32 x 32 tiles; one warp (a block of its
// own) owns a tile in shared memory with a one-node halo and runs directional
// Gauss-Seidel sweeps inside it, one anti-diagonal per step (the 32 lanes
// update the nodes of a diagonal together; they depend only on the previous
// diagonal).  A pass runs every tile whose own values or a neighbour tile's
// changed in the previous pass and writes its interior back; passes repeat
// until no value decreases by more than tol.  Tiles read their halo from
// global memory while neighbours may be writing it: any value read is an
// upper bound of the fixed point, so the monotone iteration is unaffected,
// and a tile whose neighbour changed runs again in the next pass.
//
// What bounds it: the dependent updates along the front (n / 2 diagonals or
// more from the source to the far corner, each a chain of FP64 operations of
// ~32 ns and a square root); neither bandwidth nor the number of tiles.  So a
// visit does only the sweeps that can change something: the nodes that would
// decrease (at first only the tile's edge nodes can, after a sweep all are
// looked at, which is a pipelined pass and not a chain) vote for the ordering
// their information comes from, the ordering with most
// votes is swept, and so on until no node votes.  Mostly that is one sweep
// where four orderings, twice, were swept before; the chain of an update is
// shortened by integer comparisons, one fused multiply-add per sum and a
// Goldschmidt square root, and nothing is read from global memory inside it.
// n = 2047, layered medium: 738 -> 130 us per pass, 60.0 -> 10.4 ms per call.
#include <cuda_runtime.h>

#include <cmath>
#include <string>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "handle.h"

namespace wadr {

constexpr int ET = 32;          // tile side (nodes)
constexpr int EBATCH = 8;       // passes between two looks of the host
constexpr int EMAXS = 32;       // sweeps of one visit; a tile that needs more goes on in the next pass
constexpr double EINF = 1e300;

// The nodes fixed by the source: within r_init of (x0, y0), inside the index
// box [i0, i1] x [j0, j1] (a margin of one node around the disc), at
// s0 |x - x0|, s0 = s at node (is, js).
struct EikSrc {
    double x0, y0, r_init;
    int i0, i1, j0, j1;
    int is, js;
};

// distance of node (i, j) from the source, products and sums rounded
// separately (no contraction), as the host generator and the oracle evaluate
// them
__device__ __forceinline__ double src_dist(const EikSrc& c, double h, int i, int j) {
    const double dx = __dsub_rn(__dmul_rn((double)(i + 1), h), c.x0);
    const double dy = __dsub_rn(__dmul_rn((double)(j + 1), h), c.y0);
    return sqrt(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
}
__device__ __forceinline__ bool in_box(const EikSrc& c, int i, int j) {
    return i >= c.i0 && i <= c.i1 && j >= c.j0 && j <= c.j1;
}

// tau = s(x0) |x - x0| on the fixed nodes, inf elsewhere (a plain fill: the
// distance is formed inside the box only; with a square root per node the
// FP64 pipes took 154 us at n = 2047)
__global__ void k_eik_init(int n, int ny, double h, const double* __restrict__ s, EikSrc c, double* __restrict__ tau) {
    const long long N = (long long)n * ny;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < N; p += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(p % n), j = (int)(p / n);
        double v = EINF;
        if (in_box(c, i, j)) {
            const double r = src_dist(c, h, i, j);
            if (r <= c.r_init) v = __dmul_rn(s[(long long)c.js * n + c.is], r);
        }
        tau[p] = v;
    }
}

// Square root of a normal x well inside the exponent range: Goldschmidt's
// coupled iteration from an approximate reciprocal square root (~20 bits,
// squared once), then one correction by the residual x - g^2 (as many bits
// again as the seed has): five dependent operations after the seed.
__device__ __forceinline__ double sqrt_gs(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double h = __longlong_as_double(__double_as_longlong(y) - (1ll << 52));   // y / 2
    double g = x * y;
    g = fma(g, fma(-g, h, 0.5), g);
    return fma(fma(-g, g, x), h, g);
}

// Order of two values.  FAST: both are >= 0 (or +inf, NaN last), where
// doubles order like their bits and an integer comparison takes a few
// instructions; else the FP64 comparison.
template <bool FAST> __device__ __forceinline__ bool dlt(double a, double b) {
    return FAST ? __double_as_longlong(a) < __double_as_longlong(b) : a < b;
}
template <bool FAST> __device__ __forceinline__ double dmin2(double a, double b) { return dlt<FAST>(b, a) ? b : a; }

// Godunov update from the smaller neighbour in x (a) and in y (b), f = s h,
// r0 = 2 f^2: m + f with m = min(a, b) where |a - b| >= f (also with an
// infinite neighbour), else m + (|a - b| + sqrt(r0 - (a - b)^2)) / 2.  A warp's
// FP64 instruction holds its scheduler's pipe for 64 cycles, so their number
// counts: nine here, without branches so that independent updates overlap.
// FAST: values >= 0 and f inside the range of sqrt_gs.
template <bool FAST> __device__ __forceinline__ double godunov_upd(double a, double b, double f, double r0) {
    const double d = fabs(a - b), m = dmin2<FAST>(a, b), rad = fma(-d, d, r0);
    const double two = d + (FAST ? sqrt_gs(rad) : sqrt(rad));
    // twice f: an exponent step (FAST: f is normal)
    const double one = FAST ? __longlong_as_double(__double_as_longlong(f) + (1ll << 52)) : f + f;
    return fma(0.5, dlt<FAST>(d, f) ? two : one, m);
}

// One pass over the active tiles (see the file comment).  act_in[t] != 0:
// tile t changed in the previous pass (2: all its nodes are to be looked at);
// act_out[t] is set when it changes in this one and *nchanged counts such
// tiles; act_clr is the next pass's act_out.
__global__ void __launch_bounds__(32) k_eik_pass(int n, int ny, double h, const double* __restrict__ s, EikSrc src,
                                                 double* tau, const unsigned char* __restrict__ act_in,
                                                 unsigned char* __restrict__ act_out,
                                                 unsigned char* __restrict__ act_clr, unsigned* nchanged, double tol) {
    // odd distances between the nodes of a diagonal (in 8-byte banks): no conflicts
    __shared__ double T[ET + 2][ET + 2];
    __shared__ double Fs[ET][ET], Rs[ET][ET];
    const int lane = threadIdx.x;
    const int ntx = (n + ET - 1) / ET, nty = (ny + ET - 1) / ET;
    for (int t = blockIdx.x; t < ntx * nty; t += gridDim.x) {
        const int tx = t % ntx, ty = t / ntx;
        const int self = act_in[t];
        const bool active = self || (tx > 0 && act_in[t - 1]) || (tx < ntx - 1 && act_in[t + 1]) ||
                            (ty > 0 && act_in[t - ntx]) || (ty < nty - 1 && act_in[t + ntx]);
        if (lane == 0) act_clr[t] = 0;
        if (!active) continue;                      // warp-uniform
        const int gx0 = tx * ET, gy0 = ty * ET;
        auto G = [&](int gi, int gj) -> double {
            return (gi >= 0 && gi < n && gj >= 0 && gj < ny) ? __ldcg(&tau[(long long)gj * n + gi]) : EINF;
        };
        // interior and halo rows (lane = column), halo columns (lane = row);
        // upd: the column's nodes that are in the grid and not fixed
        unsigned upd = 0;
#pragma unroll 8
        for (int r = -1; r <= ET; ++r) T[r + 1][lane + 1] = G(gx0 + lane, gy0 + r);
        T[lane + 1][0] = G(gx0 - 1, gy0 + lane);
        T[lane + 1][ET + 1] = G(gx0 + ET, gy0 + lane);
        const bool near = gx0 <= src.i1 && gx0 + ET > src.i0 && gy0 <= src.j1 && gy0 + ET > src.j0;
#pragma unroll 8
        for (int r = 0; r < ET; ++r) {
            const int gi = gx0 + lane, gj = gy0 + r;
            const bool in = gi < n && gj < ny;
            const double f = in ? __dmul_rn(__ldg(&s[(long long)gj * n + gi]), h) : 0.0;
            Fs[r][lane] = f;
            Rs[r][lane] = (f + f) * f;
            if (in) upd |= 1u << r;
        }
        if (near)
            for (int r = 0; r < ET; ++r) {
                const int gi = gx0 + lane, gj = gy0 + r;
                if (in_box(src, gi, gj) && src_dist(src, h, gi, gj) <= src.r_init) upd &= ~(1u << r);
            }
        const unsigned updr = __shfl_sync(0xffffffffu, upd, ET - 1 - lane);   // of column 31 - lane
        __syncwarp();
        // FAST: no negative value in the tile, every f between 1e-140 and 1e140
        // (by their bits).  big_hi, f_hi: upper words of the largest finite
        // value and of the largest f.
        int big_hi = 0, f_hi = 0;
        const int inf_hi = __double2hiint(EINF);
        auto top = [&](double v) {
            const int b = __double2hiint(v);
            if (b < inf_hi) big_hi = max(big_hi, b);
        };
        top(T[0][lane + 1]);
        top(T[ET + 1][lane + 1]);
        top(T[lane + 1][0]);
        top(T[lane + 1][ET + 1]);
        const long long fl = __double_as_longlong(1e-140), fh = __double_as_longlong(1e140);
        long long neg = __double_as_longlong(T[0][lane + 1]) | __double_as_longlong(T[ET + 1][lane + 1]) |
                        __double_as_longlong(T[lane + 1][0]) | __double_as_longlong(T[lane + 1][ET + 1]);
        bool fast = true;
#pragma unroll 8
        for (int r = 0; r < ET; ++r) {
            const long long f = __double_as_longlong(Fs[r][lane]);
            neg |= __double_as_longlong(T[r + 1][lane + 1]);
            top(T[r + 1][lane + 1]);
            f_hi = max(f_hi, __double2hiint(Fs[r][lane]));
            fast = fast && (!((upd >> r) & 1) || (f > fl && f < fh));
        }
        fast = __all_sync(0xffffffffu, fast && neg >= 0);
        // tol covers two units in the last place of every value this visit
        // can form (at most the largest finite one and f at every node)
        const double most = __hiloint2double(__reduce_max_sync(0xffffffffu, big_hi) + 1, 0) +
                            ET * ET * __hiloint2double(__reduce_max_sync(0xffffffffu, f_hi) + 1, 0);
        const bool ulps = tol >= 4.5e-16 * most;
        unsigned left;
        auto visit = [&](auto fc) -> bool {
            constexpr bool FAST = decltype(fc)::value;
            // the nodes that would decrease, by the ordering their information
            // comes from (bit 0 of the index: from the east, bit 1: from the
            // north): vote[q] has bit j for row j of the lane's column.  A
            // decrease that rounding alone can make (two units in the last
            // place) does not vote unless it exceeds tol; one above tol makes
            // the tile a changed one (big, looked for until it is known; from
            // then on two units are compared as integers where tol covers
            // them, ulps).
            unsigned vote[4] = {0, 0, 0, 0};
            bool big = false, known = false;
            // ordering (0..3) of node (i, j)'s vote, or -1
            auto look = [&](int i, int j, bool ok) -> int {
                const double w = T[j + 1][i], e = T[j + 1][i + 2], so = T[j][i + 1], no = T[j + 2][i + 1];
                const bool fe = dlt<FAST>(e, w), fn = dlt<FAST>(no, so);
                const double a = fe ? e : w, b = fn ? no : so;
                const double cur = T[j + 1][i + 1], v = godunov_upd<FAST>(a, b, Fs[j][i], Rs[j][i]);
                ok = ok && dlt<FAST>(dmin2<FAST>(a, b), EINF) && dlt<FAST>(v, cur);
                bool yes;
                if (FAST && known) {
                    yes = ok && __double_as_longlong(cur) - __double_as_longlong(v) > 2;
                } else {
                    const double dec = cur - v;
                    const bool over = ok && (cur >= EINF || dec > tol);
                    big = big || over;
                    yes = over || (ok && dec > 4.5e-16 * fabs(cur));
                }
                return yes ? (fe ? 1 : 0) + (fn ? 2 : 0) : -1;
            };
            auto look_all = [&]() {
                known = known && ulps;   // every decrease above tol votes
#pragma unroll 8
                for (int r = 0; r < ET; ++r) {
                    const int o = look(lane, r, (upd >> r) & 1);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (o == q) vote[q] |= 1u << r;
                }
            };
            if (self == 2) {
                look_all();
            } else {
                // the interior was at rest for the halo of its last visit
                const unsigned c0 = __shfl_sync(0xffffffffu, upd, 0), c1 = __shfl_sync(0xffffffffu, upd, ET - 1);
                const int s0 = look(lane, 0, upd & 1), s1 = look(lane, ET - 1, upd >> (ET - 1));
                const int w0 = look(0, lane, (c0 >> lane) & 1), w1 = look(ET - 1, lane, (c1 >> lane) & 1);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (s0 == q) vote[q] |= 1u;
                    if (s1 == q) vote[q] |= 1u << (ET - 1);
                    const unsigned b0 = __ballot_sync(0xffffffffu, w0 == q), b1 = __ballot_sync(0xffffffffu, w1 == q);
                    if (lane == 0) vote[q] |= b0;
                    if (lane == ET - 1) vote[q] |= b1;
                }
            }
            bool swept = false;
            int n_left = EMAXS;
            while (true) {
                known = __any_sync(0xffffffffu, big);
                // ordering with most votes over the warp (at most 1024 each)
                const unsigned lo = __reduce_add_sync(0xffffffffu, __popc(vote[0]) | (unsigned)__popc(vote[1]) << 16);
                const unsigned hi = __reduce_add_sync(0xffffffffu, __popc(vote[2]) | (unsigned)__popc(vote[3]) << 16);
                left = lo | hi;
                if (left == 0 || n_left == 0) break;
                const unsigned c[4] = {lo & 0xffffu, lo >> 16, hi & 0xffffu, hi >> 16};
                int dir = 0;
                unsigned most = c[0], vm = vote[0];
#pragma unroll
                for (int q = 1; q < 4; ++q)
                    if (c[q] > most) { most = c[q]; dir = q; vm = vote[q]; }
                const bool fwx = (dir & 1) == 0, fwy = (dir & 2) == 0;
                const unsigned um = fwx ? upd : updr;
                const int i = fwx ? lane : ET - 1 - lane;
                // the diagonals of its first and last vote: nothing changes
                // before the first, nor after the last once a few diagonals
                // in a row changed nothing
                const int ul = i;   // (lane of column `lane` in the sweep's order)
                const int first = vm ? ul + (fwy ? __ffs((int)vm) - 1 : __clz((int)vm)) : 2 * ET;
                const int last = vm ? ul + (fwy ? 31 - __clz((int)vm) : 32 - __ffs((int)vm)) : 0;
                const int u0 = (int)__reduce_min_sync(0xffffffffu, (unsigned)first);
                const int u1 = (int)__reduce_max_sync(0xffffffffu, (unsigned)last);
                bool moved = false;
                for (int u = u0; u < 2 * ET - 1; ++u) {
                    const int jj = u - lane, j = fwy ? jj : ET - 1 - jj;
                    if ((unsigned)jj < (unsigned)ET && ((um >> j) & 1)) {
                        const double a = dmin2<FAST>(T[j + 1][i], T[j + 1][i + 2]);
                        const double b = dmin2<FAST>(T[j][i + 1], T[j + 2][i + 1]);
                        const double v = godunov_upd<FAST>(a, b, Fs[j][i], Rs[j][i]);
                        if (dlt<FAST>(dmin2<FAST>(a, b), EINF) && dlt<FAST>(v, T[j + 1][i + 1])) {
                            T[j + 1][i + 1] = v;
                            moved = true;
                        }
                    }
                    __syncwarp();
                    if ((u & 3) == 3) {
                        if (!__any_sync(0xffffffffu, moved) && u >= u1) break;
                        moved = false;
                    }
                }
                swept = true;
                --n_left;
                vote[0] = vote[1] = vote[2] = vote[3] = 0;
                look_all();
            }
            // below-tol decreases are written but do not wake the neighbours
            if (swept && lane == 0 && (known || left)) {
                act_out[t] = left ? 2 : 1;
                atomicAdd(nchanged, 1u);
            }
            return swept;
        };
        const bool swept = fast ? visit(std::true_type{}) : visit(std::false_type{});
        if (swept) {
            for (int r = 0; r < ET; ++r)
                if ((upd >> r) & 1) __stcg(&tau[(long long)(gy0 + r) * n + gx0 + lane], T[r + 1][lane + 1]);
        }
        __syncwarp();
    }
}

}  // namespace wadr

using namespace wadr;

extern "C" int mg_eikonal_rect(int n, int ny, const double* s, double x0, double y0, double r_init, double tol,
                               int max_passes, double* tau, int* passes, void* stream) {
    if (n < 2 || n > 65535 || ny < 2 || ny > 65535 || !s || !tau || !(r_init >= 0) || !(tol >= 0) ||
        max_passes < 1 || !std::isfinite(x0) || !std::isfinite(y0)) {
        set_error("mg_eikonal: bad argument");
        return MG_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const double h = 1.0 / (std::max(n, ny) + 1);
    // s(x0) is taken at the node nearest to the source (per-axis rounding,
    // clamped: the nearest node of a regular grid); the fixed disc must
    // contain a node, as the host generator requires, and the nearest node is
    // the one to test
    int i0 = (int)std::floor(x0 / h - 1.0 + 0.5), j0 = (int)std::floor(y0 / h - 1.0 + 0.5);
    i0 = std::min(std::max(i0, 0), n - 1);
    j0 = std::min(std::max(j0, 0), ny - 1);
    {
        const double dx = (i0 + 1) * h - x0, dy = (j0 + 1) * h - y0;
        if (!(std::sqrt(dx * dx + dy * dy) <= r_init)) {
            set_error("mg_eikonal: no grid node within r_init of the source");
            return MG_EINVAL;
        }
    }
    const size_t N = (size_t)n * ny;
    const int ntx = (n + ET - 1) / ET, ntiles = ntx * ((ny + ET - 1) / ET);
    auto is_dev = [](const void* q) {
        cudaPointerAttributes a;
        const bool d = cudaPointerGetAttributes(&a, q) == cudaSuccess &&
                       (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged);
        cudaGetLastError();
        return d;
    };
    std::vector<void*> mine;
    auto release = [&]() { for (void* q : mine) cudaFree(q); };
    auto dalloc = [&](size_t bytes) -> void* {
        void* q = nullptr;
        if (cudaMalloc(&q, bytes) != cudaSuccess) return nullptr;
        mine.push_back(q);
        return q;
    };
    const double* ds = s;
    if (!is_dev(s)) {
        double* q = (double*)dalloc(N * 8);
        if (!q) { release(); set_error("mg_eikonal: out of device memory"); return MG_ENOMEM; }
        cudaMemcpyAsync(q, s, N * 8, cudaMemcpyHostToDevice, st);
        ds = q;
    }
    double* dt = is_dev(tau) ? tau : (double*)dalloc(N * 8);
    // three activity tables (read, written, cleared for the pass after) and
    // the changed-tile counts of a batch of passes
    unsigned char* act = (unsigned char*)dalloc(3 * (size_t)ntiles + 256 + EBATCH * sizeof(unsigned));
    if (!dt || !act) {
        release();
        set_error("mg_eikonal: out of device memory");
        return MG_ENOMEM;
    }
    unsigned* cnt = (unsigned*)(((uintptr_t)(act + 3 * (size_t)ntiles) + 255) / 256 * 256);
    EikSrc src;
    src.x0 = x0;
    src.y0 = y0;
    src.r_init = r_init;
    src.is = i0;
    src.js = j0;
    {
        // index box of the fixed disc, one node wider on every side
        auto lo = [&](double c) { return (int)std::max(-1.0, std::min((c - r_init) / h - 3.0, 65536.0)); };
        auto hi = [&](double c) { return (int)std::max(-1.0, std::min((c + r_init) / h + 2.0, 65536.0)); };
        src.i0 = lo(x0);
        src.i1 = hi(x0);
        src.j0 = lo(y0);
        src.j1 = hi(y0);
    }
    k_eik_init<<<1216, 256, 0, st>>>(n, ny, h, ds, src, dt);
    cudaMemsetAsync(act, 2, (size_t)ntiles, st);            // every tile is looked at in the first pass
    cudaMemsetAsync(act + ntiles, 0, 2 * (size_t)ntiles, st);
    const unsigned nblk = (unsigned)std::min(ntiles, 16384);
    int pass = 0, rc = MG_ENOTCONV;
    unsigned hcnt[EBATCH];
    while (pass < max_passes && rc != MG_OK) {
        // a few passes per look of the host: after the pass that changed
        // nothing the rest of a batch finds no active tile
        const int nb = std::min(EBATCH, max_passes - pass);
        cudaMemsetAsync(cnt, 0, EBATCH * sizeof(unsigned), st);
        for (int q = 0; q < nb; ++q) {
            unsigned char* a_in = act + (size_t)((pass + q) % 3) * ntiles;
            unsigned char* a_out = act + (size_t)((pass + q + 1) % 3) * ntiles;
            unsigned char* a_clr = act + (size_t)((pass + q + 2) % 3) * ntiles;
            k_eik_pass<<<nblk, 32, 0, st>>>(n, ny, h, ds, src, dt, a_in, a_out, a_clr, cnt + q, tol);
        }
        cudaMemcpyAsync(hcnt, cnt, sizeof(unsigned) * nb, cudaMemcpyDeviceToHost, st);
        cudaError_t e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) {
            release();
            set_error(std::string("mg_eikonal: ") + cudaGetErrorString(e));
            return MG_ECUDA;
        }
        for (int q = 0; q < nb; ++q) {
            ++pass;
            if (hcnt[q] == 0) {
                rc = MG_OK;
                break;
            }
        }
    }
    if (dt != tau) cudaMemcpyAsync(tau, dt, N * 8, cudaMemcpyDeviceToHost, st);
    cudaError_t e = cudaStreamSynchronize(st);
    release();
    if (e != cudaSuccess) {
        set_error(std::string("mg_eikonal: ") + cudaGetErrorString(e));
        return MG_ECUDA;
    }
    if (passes) *passes = pass;
    if (rc != MG_OK) set_error("mg_eikonal: max_passes reached before no value changed by more than tol");
    return rc;
}

extern "C" int mg_eikonal(int n, const double* s, double x0, double y0, double r_init, double tol, int max_passes,
                          double* tau, int* passes, void* stream) {
    return mg_eikonal_rect(n, n, s, x0, y0, r_init, tol, max_passes, tau, passes, stream);
}
