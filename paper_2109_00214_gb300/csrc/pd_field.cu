// pd_field.cu -- Poisson solve of Eq. (8), read as lap(phi) = -rho/eps0, on the
// r-z node grid of every run, and E = -grad(phi).
//
// Discretisation (finite volumes around each node (i, j)):
//   ap_j (phi_{j+1} - phi_j) + am_j (phi_{j-1} - phi_j)
//     + b_j (phi_{i+1} - 2 phi_i + phi_{i-1}) = -rho_ij Vfv_j / eps0
// with ap_j = 2 pi r_{j+1/2} dz/dr (0 at r = R), am_j = 2 pi r_{j-1/2} dz/dr (0
// on the axis), b_j = A_j / dz, A_j the area of the node's radial extent and
// Vfv_j = A_j dz.  The node density rho_ij = Q_ij / V_ij uses Verboncoeur's
// volumes.  phi = 0 on the cathode row, V on the anode row.  In matrix form
// A phi = b on the interior rows.
//
// Solver: defect correction in double precision around a single-precision
// multigrid.  Each cycle takes the residual r = b - A phi in double (with its
// norm, the convergence test), solves A e = r approximately by one float
// V(2,2) cycle from e = 0, and adds e to phi in double.  GB300 does double
// arithmetic at a small fraction of its float rate, so only the residual and
// the update are double; the cycle converges like a double one as long as
// each correction is accurate to a few digits, and phi reaches residuals far
// below float precision.
//
// V-cycle: red-black Gauss-Seidel (four half-sweeps per launch, a warp a tile
// of the grid in its registers), restriction of the integrated residuals by
// full weighting (1, 1/2, 1/4), bilinear prolongation, coefficients
// rediscretised on each level, and an exact solve on the coarsest level by its
// inverse (formed on the host once; Gauss-Seidel sweeps instead when the
// coarsest level has more than MG_DIRECT_MAX unknowns).  A level takes one
// launch on the way down (smoothing, residual and restriction), one on the way
// up (prolongation and smoothing); the levels of at most 2048 nodes take one
// launch together, and the residual with its norm the last of a cycle.
//
// Batched over runs: the per-cycle kernels take work lists of (run, tile) per
// level, so a launch has only warps with work; a run that has
// converged skips the rest of the cycles.  Per-run residual norms and
// converged flags stay on the device.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "pd_field.h"

namespace pd {

namespace {
constexpr double QE_ = 1.602176634e-19;
constexpr double EPS0_ = 8.8541878128e-12;
constexpr double PI_ = 3.14159265358979323846;
constexpr int RED_ROWS = 4;            // a warp's part of the residual: 32 radial nodes x 4 rows
constexpr int RED_WARPS = 4;           // of a block
constexpr int TILE_WARPS = 4;          // tiles of a block of the smoothing kernels
// A smoothing tile is a window of 64 radial nodes x K rows, two columns to a
// lane and the rows in registers; each half-sweep spoils a ring of the window,
// so a tile gives the window less 4 nodes a side (post-smoothing), or less 6
// (pre-smoothing, whose restriction reads two nodes further).
constexpr int WIN_C = 64, PRE_H = 6, POST_H = 4;
constexpr int K_SMALL = 20, K_LARGE = 32;
constexpr int SMALL_TILES = 4 * 152;   // long windows from this many tiles on
// Levels from the first one with at most this many nodes (two of a color a thread):
// k_mg_tail.  A level there takes 3-4 us of a cycle, its two launches 11: from 1156
// nodes on, 224 x 96 cells 3.74 -> 3.65 ms, 448 x 256 3.15 -> 3.02 (57 x 25 and 57 x
// 33 nodes).
constexpr int TAIL_NODES = 2048;
constexpr int TAIL_THREADS = 512;
constexpr int TAIL_SLOTS = 2;          // nodes of a color a thread of k_mg_tail holds (most levels: one)
// Dynamic shared memory k_mg_tail may take: levels of up to 2048 nodes 24 KB, the
// coarser ones a third of that, their coefficients, an inverse 40 KB at most; the
// most of any grid is 73.7 KB (160 x 768 cells, from 40 x 192 of them on).
constexpr size_t TAIL_SMEM_MAX = 80 * 1024;

size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

void level_dims(int nz, int nr, int* nzs, int* nrs, int& nlev) {
    nzs[0] = nz;
    nrs[0] = nr;
    nlev = 1;
    while (nlev < MG_MAX_LEVELS && nzs[nlev - 1] % 2 == 0 && nrs[nlev - 1] % 2 == 0 && nzs[nlev - 1] > 8 &&
           nrs[nlev - 1] > 8) {
        nzs[nlev] = nzs[nlev - 1] / 2;
        nrs[nlev] = nrs[nlev - 1] / 2;
        ++nlev;
    }
}

// unknowns of the coarsest level (interior rows, all radial nodes)
int coarse_unknowns(const int* a, const int* b, int n) { return (a[n - 1] - 1) * (b[n - 1] + 1); }

// first level cycled by k_mg_tail (the coarsest level always qualifies: at
// most 1024 nodes)
int tail_level(const int* a, const int* b, int n) {
    for (int l = 0; l < n; ++l)
        if ((a[l] + 1) * (b[l] + 1) <= TAIL_NODES && (a[l] - 1) * ((b[l] + 2) / 2) <= TAIL_SLOTS * TAIL_THREADS) return l;
    return n - 1;
}

int tiles_of(int nz, int nr, int K, int halo) {
    const int ti = K - 2 * halo, tj = WIN_C - 2 * halo;
    return ((nz + ti - 1) / ti) * ((nr + tj) / tj);
}
int red_units(int nz, int nr) { return ((nz - 1 + RED_ROWS - 1) / RED_ROWS) * ((nr + 32) / 32); }
int red_blocks(int nz, int nr) { return (red_units(nz, nr) + RED_WARPS - 1) / RED_WARPS; }

// work-list entries of one run (all levels that smooth)
size_t run_tasks(int nz, int nr) {
    int a[MG_MAX_LEVELS], b[MG_MAX_LEVELS], n;
    level_dims(nz, nr, a, b, n);
    size_t t = 0;
    for (int l = 0; l + 1 < n; ++l)
        t += tiles_of(a[l], b[l], K_SMALL, PRE_H) + tiles_of(a[l], b[l], K_SMALL, POST_H);
    return t + red_blocks(nz, nr);
}

// device bytes of one run, in the order field_init takes them
size_t run_bytes(int nz, int nr) {
    int a[MG_MAX_LEVELS], b[MG_MAX_LEVELS], n;
    level_dims(nz, nr, a, b, n);
    const size_t W0 = (size_t)nr + 1, nodes0 = ((size_t)nz + 1) * W0;
    size_t t = al(nodes0 * 8) + 6 * al(W0 * 8);            // b, and ap, am, b, dg, cr, iv of level 0 in double
    for (int l = 0; l < n; ++l) {
        const size_t W = (size_t)b[l] + 1, nodes = ((size_t)a[l] + 1) * W;
        t += 3 * al(nodes * 4) + 4 * al(W * 4);             // e, e2, f; ap, am, b, dinv in float
    }
    for (int l = tail_level(a, b, n); l < n; ++l) t += al(4 * ((size_t)b[l] + 1) * 4);   // k_mg_tail's coefficients
    const size_t m = (size_t)coarse_unknowns(a, b, n);
    if (m <= (size_t)MG_DIRECT_MAX) t += al(m * m * 4 + 16);            // (read in units of 16 bytes)
    return t;
}
}  // namespace

bool field_grid_ok(int nz, int nr) {
    int a[MG_MAX_LEVELS], b[MG_MAX_LEVELS], n;
    level_dims(nz, nr, a, b, n);
    return (a[n - 1] + 1) * (b[n - 1] + 1) <= 1024 && a[n - 1] >= 2 && b[n - 1] >= 2;
}

size_t field_workspace_bytes(const std::vector<int>& nz, const std::vector<int>& nr) {
    size_t t = 0;
    const size_t R = nz.size();
    size_t tasks = 0, red = 0;
    for (size_t r = 0; r < R; ++r) {
        t += run_bytes(nz[r], nr[r]);
        tasks += run_tasks(nz[r], nr[r]);
        red += red_blocks(nz[r], nr[r]);
    }
    t += al(R * MG_MAX_LEVELS * sizeof(MGLevel)) + al(R * sizeof(MGTop)) + al(R * 4) * 3 +
         al(red * 2 * 8) + al(R * 8) * 2 + al(R * sizeof(TailRun)) + al(tasks * sizeof(int2) + 8);
    return t;
}

// ------------------------------------------------------------------
// kernels
// ------------------------------------------------------------------
// The residual r = b - A phi of every run in double, its norm (and, on the
// first of a solve, that of b), and the right-hand side of the next correction:
// level 0's f = r (float).  A warp takes 32 radial nodes and marches over
// RED_ROWS rows, so that each node of phi is read once a row, not three times;
// double arithmetic (seven operations a node) bounds it, and small units spread it
// over the SMs: 120 x 480 cells 11.8 us with 8 rows a warp and 8 warps a block, 8.8
// now.  Work list of (run, first unit), four units a block; the block that finishes
// a run's last units sums the blocks' parts in their order and judges the run:
// relres = |r| / |b|, converged flag, bookkeeping.
// 512 x 512 cells, device time of a launch under ncu: 14.7 us with the norm (13.8
// + 8.9 us as a launch of rows and one of norms).
__global__ void __launch_bounds__(32 * RED_WARPS) k_residual_norms(const MGTop* top, const MGLevel* lev, const int2* tasks,
                                                        const int* red_base, double* red, unsigned int* ticket,
                                                        double* bnorm, int* done, const double* tol, RunState* rs,
                                                        int cycle, MGTop one, float* one_f) {
    const int2 tk = tasks ? tasks[blockIdx.x] : make_int2(0, (int)blockIdx.x * RED_WARPS);
    const int run = tk.x;
    const int skip = cycle > 0 ? done[run] : 0;
    const MGTop T = tasks ? top[run] : one;
    const int nz = T.nz, nr = T.nr, W = nr + 1;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int cols = (W + 31) / 32, rows = (nz - 1 + RED_ROWS - 1) / RED_ROWS;
    const int u = tk.y + w;
    double acc = 0.0, accb = 0.0;
    if (u < cols * rows) {
        const int j = (u % cols) * 32 + lane, i0 = 1 + (u / cols) * RED_ROWS, i1 = min(i0 + RED_ROWS, nz);
        if (j < W) {
            const double *x = T.phi, *bf = T.bf;
            float* f = tasks ? lev[run * MG_MAX_LEVELS].f : one_f;
            const double dg = T.dg[j], ap = T.ap[j], am = T.am[j], bz = T.b[j];
            // every load before the first use: their latencies overlap
            double xc[RED_ROWS + 2], xp[RED_ROWS], xm[RED_ROWS], bk[RED_ROWS];
            const int rt = j < nr ? 1 : 0, lf = j > 0 ? 1 : 0;
#pragma unroll
            for (int q = 0; q < RED_ROWS + 2; ++q) {
                const int i = min(i0 - 1 + q, nz);
                xc[q] = x[i * W + j];
            }
#pragma unroll
            for (int q = 0; q < RED_ROWS; ++q) {
                const int k = min(i0 + q, nz) * W + j;
                xp[q] = x[k + rt];
                xm[q] = x[k - lf];
                bk[q] = bf[k];
            }
            if (skip) return;
#pragma unroll
            for (int q = 0; q < RED_ROWS; ++q) {
                const int i = i0 + q;
                if (i < i1) {
                    const double xu = i + 1 < nz ? xc[q + 2] : 0.0;      // the anode row is in b
                    const double xd = i - 1 > 0 ? xc[q] : 0.0;
                    double r = bk[q] - dg * xc[q + 1];
                    r += ap * xp[q];                                     // ap = 0 on the last column
                    r += am * xm[q];                                     // am = 0 on the axis
                    r += bz * (xu + xd);
                    f[i * W + j] = (float)r;
                    acc += r * r;
                    if (cycle == 0) accb += bk[q] * bk[q];
                }
            }
        }
    }
    if (skip) return;                                  // (the same for the whole block)
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
        accb += __shfl_down_sync(0xFFFFFFFFu, accb, o);
    }
    __shared__ double sa[RED_WARPS], sb[RED_WARPS];
    __shared__ bool s_last;
    if (lane == 0) {
        sa[w] = acc;
        sb[w] = accb;
    }
    __syncthreads();
    const int blocks = (cols * rows + RED_WARPS - 1) / RED_WARPS;
    double* rd = red + 2 * (size_t)red_base[run];
    if (threadIdx.x == 0) {
        double t = 0, tb = 0;
        for (int q = 0; q < RED_WARPS; ++q) {
            t += sa[q];
            tb += sb[q];
        }
        __stcg(&rd[2 * (tk.y / RED_WARPS)], t);
        __stcg(&rd[2 * (tk.y / RED_WARPS) + 1], tb);
        __threadfence();
        s_last = atomicAdd(&ticket[run], 1u) == (unsigned int)(blocks - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    acc = accb = 0.0;
    for (int q = threadIdx.x; q < blocks; q += 32 * RED_WARPS) {
        acc += __ldcg(&rd[2 * q]);
        accb += __ldcg(&rd[2 * q + 1]);
    }
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
        accb += __shfl_down_sync(0xFFFFFFFFu, accb, o);
    }
    if (lane == 0) {
        sa[w] = acc;
        sb[w] = accb;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    double a = 0, b = 0;
    for (int q = 0; q < RED_WARPS; ++q) {
        a += sa[q];
        b += sb[q];
    }
    ticket[run] = 0u;
    const double rn = sqrt(a);
    if (cycle == 0) bnorm[run] = sqrt(b);
    const double bn = bnorm[run];
    const double rel = bn > 0 ? rn / bn : 0.0;
    rs[run].relres = rel;
    rs[run].cycles = (double)cycle;
    if (cycle == 0) rs[run].relres0 = rel;
    int d = 0;
    if (!(rel == rel) || !(bn == bn)) d = 2;              // non-finite: stop this run
    else if (bn == 0.0 || rel <= tol[run]) d = 1;
    done[run] = d;
}

// The window of a warp's tile: two columns a lane (j = j0 + 2 lane and the next),
// K rows from i0, both even, so that which of a lane's columns has a color
// follows from the row's number alone.
template <int K>
struct Window {
    float x0[K], x1[K], f0[K], f1[K];
    float ap0, am0, b0, d0, ap1, am1, b1, d1;
};

// the coefficients of the lane's columns (zero outside the grid: such nodes stay
// zero) and the right-hand side
template <int K>
__device__ __forceinline__ void window_load(Window<K>& w, const MGLevel& L, int i0, int j) {
    const int W = L.nr + 1;
    const bool in0 = j >= 0 && j <= L.nr, in1 = j + 1 >= 0 && j + 1 <= L.nr;
    w.ap0 = in0 ? L.ap[j] : 0.0f;
    w.am0 = in0 ? L.am[j] : 0.0f;
    w.b0 = in0 ? L.b[j] : 0.0f;
    w.d0 = in0 ? L.dinv[j] : 0.0f;
    w.ap1 = in1 ? L.ap[j + 1] : 0.0f;
    w.am1 = in1 ? L.am[j + 1] : 0.0f;
    w.b1 = in1 ? L.b[j + 1] : 0.0f;
    w.d1 = in1 ? L.dinv[j + 1] : 0.0f;
    const float* f = L.f;
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int i = i0 + r;
        const bool in = i >= 1 && i <= L.nz - 1;
        const int k = i * W + j;
        w.f0[r] = in && in0 ? f[k] : 0.0f;
        w.f1[r] = in && in1 ? f[k + 1] : 0.0f;
    }
}

// One half-sweep of red-black Gauss-Seidel on A e = f: the nodes with (i + j) & 1
// == C.  Rows outside the grid stay zero.
template <int K, int C>
__device__ __forceinline__ void window_sweep(Window<K>& w, int i0, int nz) {
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const bool in = i0 + r >= 1 && i0 + r <= nz - 1;
        if (((C + r) & 1) == 0) {
            const float xl = __shfl_up_sync(0xFFFFFFFFu, w.x1[r], 1);
            float v = w.f0[r];
            v = fmaf(w.ap0, w.x1[r], v);
            v = fmaf(w.am0, xl, v);
            if (r + 1 < K) v = fmaf(w.b0, w.x0[r + 1 < K ? r + 1 : r], v);
            if (r > 0) v = fmaf(w.b0, w.x0[r > 0 ? r - 1 : r], v);
            w.x0[r] = in ? v * w.d0 : 0.0f;
        } else {
            const float xr = __shfl_down_sync(0xFFFFFFFFu, w.x0[r], 1);
            float v = w.f1[r];
            v = fmaf(w.ap1, xr, v);
            v = fmaf(w.am1, w.x0[r], v);
            if (r + 1 < K) v = fmaf(w.b1, w.x1[r + 1 < K ? r + 1 : r], v);
            if (r > 0) v = fmaf(w.b1, w.x1[r > 0 ? r - 1 : r], v);
            w.x1[r] = in ? v * w.d1 : 0.0f;
        }
    }
}

// The way down a level: four half-sweeps (colors 0, 1, 0, 1) from e = 0 into e2,
// the residual r = f - A e2, and the next level's right-hand side, the sum of
// the residuals over its control volumes (full weighting scaled by 4).  The
// window's even columns are the coarse nodes': lane = coarse column.
// Latency bounds it on one grid (all loads before the first use, no barrier).
// Average over the levels of 512 x 512 cells: 5.2 us, against 8.8 us for the
// smoothing by a block through shared memory plus 6.9 us for the restriction.
template <int K>
__global__ void __launch_bounds__(TILE_WARPS * 32, K == K_LARGE ? 3 : 4) k_down(const MGLevel* lev, const int* done, int l,
                                                          const int2* tasks, int ntask, MGLevel one) {
    constexpr int TI = K - 2 * PRE_H, TJ = WIN_C - 2 * PRE_H;
    const int t = blockIdx.x * TILE_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (t >= ntask) return;
    const int2 tk = tasks ? tasks[t] : make_int2(0, t);
    const int skip = done[tk.x];
    const MGLevel L = tasks ? lev[tk.x * MG_MAX_LEVELS + l] : one;
    const int nz = L.nz, nr = L.nr, W = nr + 1;
    const int tj = (W + TJ - 1) / TJ;
    const int i0 = (tk.y / tj) * TI - PRE_H, j0 = (tk.y % tj) * TJ - PRE_H, j = j0 + 2 * lane;
    Window<K> w;
    window_load(w, L, i0, j);
    if (skip) return;
    // color 0 from zero: f / d
#pragma unroll
    for (int r = 0; r < K; ++r) {
        w.x0[r] = (r & 1) == 0 ? w.f0[r] * w.d0 : 0.0f;
        w.x1[r] = (r & 1) == 0 ? 0.0f : w.f1[r] * w.d1;
    }
    window_sweep<K, 1>(w, i0, nz);
    window_sweep<K, 0>(w, i0, nz);
    window_sweep<K, 1>(w, i0, nz);
    {
        const bool c0 = lane >= PRE_H / 2 && lane < 32 - PRE_H / 2 && j <= nr, c1 = c0 && j + 1 <= nr;
        float* e2 = L.e2;
#pragma unroll
        for (int r = PRE_H; r < K - PRE_H; ++r) {
            const int i = i0 + r;
            if (i < 1 || i > nz - 1) continue;
            if (c0) e2[i * W + j] = w.x0[r];
            if (c1) e2[i * W + j + 1] = w.x1[r];
        }
    }
    // residuals over f (rows PRE_H - 1 .. K - PRE_H)
    const float dg0 = w.ap0 + w.am0 + 2.0f * w.b0, dg1 = w.ap1 + w.am1 + 2.0f * w.b1;
#pragma unroll
    for (int r = PRE_H - 1; r <= K - PRE_H; ++r) {
        const float xl = __shfl_up_sync(0xFFFFFFFFu, w.x1[r], 1), xr = __shfl_down_sync(0xFFFFFFFFu, w.x0[r], 1);
        float s = dg0 * w.x0[r];
        s = fmaf(-w.ap0, w.x1[r], s);
        s = fmaf(-w.am0, xl, s);
        s = fmaf(-w.b0, w.x0[r + 1], s);
        s = fmaf(-w.b0, w.x0[r - 1], s);
        w.f0[r] = w.f0[r] - s;
        s = dg1 * w.x1[r];
        s = fmaf(-w.ap1, xr, s);
        s = fmaf(-w.am1, w.x0[r], s);
        s = fmaf(-w.b1, w.x1[r + 1], s);
        s = fmaf(-w.b1, w.x1[r - 1], s);
        w.f1[r] = w.f1[r] - s;
    }
    const MGLevel& Cl = lev[tk.x * MG_MAX_LEVELS + l + 1];
    const int Wc = Cl.nr + 1, nzc = Cl.nz, J = j >> 1;
    float* cf = Cl.f;
    const bool out = lane >= PRE_H / 2 && lane < 32 - PRE_H / 2 && j <= nr;
#pragma unroll
    for (int r = PRE_H; r < K - PRE_H; r += 2) {
        const int I = (i0 + r) >> 1;
        float s = 0.0f;
#pragma unroll
        for (int di = -1; di <= 1; ++di) {
            const float wi = di == 0 ? 1.0f : 0.5f;
            const float left = __shfl_up_sync(0xFFFFFFFFu, w.f1[r + di], 1);
            s = fmaf(0.5f * wi, left, s);
            s = fmaf(wi, w.f0[r + di], s);
            s = fmaf(0.5f * wi, w.f1[r + di], s);
        }
        if (out && I >= 1 && I <= nzc - 1) cf[I * Wc + J] = s;
    }
}

// The way up a level: e2 plus the bilinear prolongation of level l + 1's
// correction (its e), four half-sweeps (colors 1, 0, 1, 0), into e, or, with
// FINAL (level 0), added to phi.  512 x 512 cells: 10.2 us on level 0 and 6.5 us on
// the others' average (16.3 and 12.9 us by a block through shared memory).
template <int K, bool FINAL>
__global__ void __launch_bounds__(TILE_WARPS * 32, K == K_LARGE ? 2 : 3) k_up(const MGLevel* lev, const MGTop* top, const int* done, int l,
                                                        const int2* tasks, int ntask, MGLevel one, MGLevel coarse,
                                                        double* one_phi) {
    constexpr int TI = K - 2 * POST_H, TJ = WIN_C - 2 * POST_H;
    const int t = blockIdx.x * TILE_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (t >= ntask) return;
    const int2 tk = tasks ? tasks[t] : make_int2(0, t);
    const int skip = done[tk.x];
    const MGLevel L = tasks ? lev[tk.x * MG_MAX_LEVELS + l] : one;
    const int nz = L.nz, nr = L.nr, W = nr + 1;
    const int tj = (W + TJ - 1) / TJ;
    const int i0 = (tk.y / tj) * TI - POST_H, j0 = (tk.y % tj) * TJ - POST_H, j = j0 + 2 * lane;
    Window<K> w;
    window_load(w, L, i0, j);
    if (skip) return;
    {
        const MGLevel Cl = tasks ? lev[tk.x * MG_MAX_LEVELS + l + 1] : coarse;
        const int Wc = Cl.nr + 1, J = j >> 1;
        const float *ce = Cl.e, *e2 = L.e2;
        const bool in0 = j >= 0 && j <= nr, in1 = j + 1 >= 1 && j + 1 <= nr;
        // coarse rows from i0 / 2 at columns J and J + 1 (those of the grid), and
        // e2: every load before the first use, so that their latencies overlap
        float a0[K / 2 + 1], a1[K / 2 + 1];
#pragma unroll
        for (int r = 0; r <= K / 2; ++r) {
            const int I = (i0 >> 1) + r;
            const bool inI = I >= 0 && I <= Cl.nz;
            a0[r] = inI && in0 ? ce[I * Wc + J] : 0.0f;
            a1[r] = inI && in1 ? ce[I * Wc + J + 1] : 0.0f;
        }
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const int i = i0 + r, k = i * W + j;
            const bool in = i >= 1 && i <= nz - 1;
            w.x0[r] = in && in0 ? e2[k] : 0.0f;
            w.x1[r] = in && in1 ? e2[k + 1] : 0.0f;
        }
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const bool in = i0 + r >= 1 && i0 + r <= nz - 1;
            const float p0 = a0[r / 2], p1 = a1[r / 2], q0 = a0[(r + 1) / 2], q1 = a1[(r + 1) / 2];
            const float s0 = ((p0 + q0) + p0) + q0, s1 = ((p0 + q0) + p1) + q1;
            w.x0[r] = in && in0 ? fmaf(0.25f, s0, w.x0[r]) : 0.0f;
            w.x1[r] = in && in1 ? fmaf(0.25f, s1, w.x1[r]) : 0.0f;
        }
    }
    window_sweep<K, 1>(w, i0, nz);
    window_sweep<K, 0>(w, i0, nz);
    window_sweep<K, 1>(w, i0, nz);
    window_sweep<K, 0>(w, i0, nz);
    const bool c0 = lane >= POST_H / 2 && lane < 32 - POST_H / 2 && j <= nr, c1 = c0 && j + 1 <= nr;
    if (FINAL) {
        double* phi = tasks ? top[tk.x].phi : one_phi;
        double p0[TI], p1[TI];
#pragma unroll
        for (int r = 0; r < TI; ++r) {
            const int i = i0 + POST_H + r, k = i * W + j;
            const bool in = i >= 1 && i <= nz - 1;
            p0[r] = in && c0 ? phi[k] : 0.0;
            p1[r] = in && c1 ? phi[k + 1] : 0.0;
        }
#pragma unroll
        for (int r = 0; r < TI; ++r) {
            const int i = i0 + POST_H + r, k = i * W + j;
            const bool in = i >= 1 && i <= nz - 1;
            if (in && c0) phi[k] = p0[r] + (double)w.x0[POST_H + r];
            if (in && c1) phi[k + 1] = p1[r] + (double)w.x1[POST_H + r];
        }
    } else {
        float* e = L.e;
#pragma unroll
        for (int r = POST_H; r < K - POST_H; ++r) {
            const int i = i0 + r;
            if (i < 1 || i > nz - 1) continue;
            if (c0) e[i * W + j] = w.x0[r];
            if (c1) e[i * W + j + 1] = w.x1[r];
        }
    }
}

// The levels of one run from its first tail level T down to its coarsest,
// one V(2,2) cycle by one block in shared memory (blockIdx.x = run): on each
// level four red-black half-sweeps (colors 0, 1, 0, 1), the residual and the
// full-weighting restriction; on the coarsest e = A^-1 f with the stored inverse
// (transposed: column v at inv[v * m]) or `sweeps` Gauss-Seidel sweeps; then
// bilinear prolongation and four half-sweeps (colors 1, 0, 1, 0) on the way up.
// Input: f of level T (its e is zero).  Output: the correction of level T in its
// e, or, when T is level 0, added to phi.
//
// A chain of short phases between block barriers bounds it, so a thread keeps
// its nodes (one of each color, two on a few narrow grids), their right-hand
// sides and coefficients in registers through a level's sweeps, and a phase is
// four shared-memory reads, five operations and a write; the run's table and
// its coefficients come in one copy each.  An inverse of up to INV_SMEM unknowns is
// copied into shared memory by cp.async meanwhile (21 KB at 8 x 8 cells; from L2,
// when it is needed, it cost 1.2 us more).  Three levels from 28 x 12 cells: 9.3
// -> 8.0 us by that; with 14 x 61 coarsest unknowns by 200 sweeps (the paper's
// domain): 156 us with the nodes in shared memory, now 25 us.
static_assert(sizeof(TailRun) / 4 <= TAIL_THREADS, "a thread a word");
constexpr int INV_SMEM = 100;          // unknowns up to which the inverse is copied into shared memory (40 KB)
constexpr int GS_DIM = 64;             // rows and radial nodes up to which the sweeps run in registers
static_assert(GS_DIM / 4 * 32 <= TAIL_THREADS && GS_DIM == 2 * 32, "four rows a warp, two columns a lane");

struct TailLevel {
    float *e, *f, *r, *ap, *am, *b, *d;
    int nz, nr;
};

struct TailNode {
    int k, up, dn;                       // node; the rows above and below (itself's zero coefficient at an electrode)
    int rt, lf;
    float f, ap, am, bu, bd, d;
};

// the thread's nodes of each color (k < 0: none)
__device__ __forceinline__ void tail_nodes(const TailLevel& L, TailNode (&nd)[2][TAIL_SLOTS]) {
    const int W = L.nr + 1, half = (W + 1) / 2, n = (L.nz - 1) * half;
#pragma unroll
    for (int q = 0; q < TAIL_SLOTS; ++q) {
        const int p = (int)threadIdx.x + q * TAIL_THREADS;
        nd[0][q].k = nd[1][q].k = -1;
        if (p >= n) continue;
        const int i = 1 + p / half, jj = 2 * (p - (i - 1) * half);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int j = jj + ((i + c) & 1);
            if (j > L.nr) continue;
            TailNode& t = nd[c][q];
            const int k = i * W + j;
            t.k = k;
            t.f = L.f[k];
            t.ap = j < L.nr ? L.ap[j] : 0.0f;
            t.am = j > 0 ? L.am[j] : 0.0f;
            t.bu = i + 1 < L.nz ? L.b[j] : 0.0f;
            t.bd = i - 1 > 0 ? L.b[j] : 0.0f;
            t.d = L.d[j];
            t.rt = j < L.nr ? k + 1 : k;
            t.lf = j > 0 ? k - 1 : k;
            t.up = k + W;
            t.dn = k - W;
        }
    }
}

__device__ __forceinline__ void tail_half_sweep(const TailLevel& L, const TailNode (&nd)[TAIL_SLOTS]) {
    float* e = L.e;
#pragma unroll
    for (int q = 0; q < TAIL_SLOTS; ++q) {
        const TailNode& t = nd[q];
        if (t.k < 0) continue;
        float v = t.f;
        v = fmaf(t.ap, e[t.rt], v);
        v = fmaf(t.am, e[t.lf], v);
        v = fmaf(t.bu, e[t.up], v);
        v = fmaf(t.bd, e[t.dn], v);
        e[t.k] = v * t.d;
    }
    __syncthreads();
}

// `sweeps` Gauss-Seidel sweeps (color 0, then 1) from zero on a grid of at most
// GS_DIM rows (the cathode's included) and radial nodes, the operations of
// tail_half_sweep.  The sweeps are a serial chain, so the nodes stay in registers:
// four rows a warp, two columns a lane; a half-sweep exchanges columns by
// shuffles and each warp's outer rows through shared memory, one barrier of the
// sweeping warps.  15 x 60 cells, 200 sweeps, whole kernel: 51 us with a node a
// thread in shared memory, 35-41 us by a single warp (no barrier; its FMAs
// bound it), 25 us.
__device__ __forceinline__ void tail_sweeps_rows(const TailLevel& L, int sweeps, int warps) {
    const int lane = threadIdx.x & 31, w = threadIdx.x / 32, W = L.nr + 1;
    __shared__ float first[GS_DIM / 4 + 2][2][32], last[GS_DIM / 4 + 2][2][32];    // rows of warp w at w + 1, by column
    float x[2][6], f[2][6], d[2][6], ap[2], am[2], b[2];        // [1 + k]: row 4 w + k
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int j = 2 * lane + c;
        const bool in = j < W;
        const float dj = in ? L.d[j] : 0.0f;
        ap[c] = j < L.nr ? L.ap[j] : 0.0f;
        am[c] = in && j > 0 ? L.am[j] : 0.0f;
        b[c] = in ? L.b[j] : 0.0f;
        x[c][0] = x[c][5] = 0.0f;
#pragma unroll
        for (int k = 1; k < 5; ++k) {
            const int i = 4 * w + k - 1;
            const bool inner = in && i >= 1 && i < L.nz;        // others stay zero
            x[c][k] = 0.0f;
            f[c][k] = inner ? L.f[i * W + j] : 0.0f;
            d[c][k] = inner ? dj : 0.0f;
        }
        if (w == 0) last[0][c][lane] = 0.0f;
        if (w == warps - 1) first[warps + 1][c][lane] = 0.0f;
    }
    // rows of parity o of the lane's column c
    auto half = [&](int c, int o) {
#pragma unroll
        for (int k = o ? 2 : 1; k < 5; k += 2) {
            const float same = x[1 - c][k];
            const float other = c ? __shfl_down_sync(0xFFFFFFFFu, same, 1) : __shfl_up_sync(0xFFFFFFFFu, same, 1);
            float v = fmaf(ap[c], c ? other : same, f[c][k]);
            v = fmaf(am[c], c ? same : other, v);
            v = fmaf(b[c], x[c][k + 1], v);
            v = fmaf(b[c], x[c][k - 1], v);
            x[c][k] = v * d[c][k];
        }
        if (o == 0) first[w + 1][c][lane] = x[c][1];
        else last[w + 1][c][lane] = x[c][4];
    };
    // the neighbours' rows, after even rows of column c and odd ones of the other
    auto meet = [&](int c) {
        asm volatile("bar.sync 1, %0;" ::"r"(32 * warps) : "memory");
        x[c][5] = first[w + 2][c][lane];
        x[1 - c][0] = last[w][1 - c][lane];
    };
#pragma unroll 1
    for (int it = 0; it < sweeps; ++it) {
        half(0, 0);
        half(1, 1);
        meet(0);
        half(1, 0);
        half(0, 1);
        meet(1);
    }
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int k = 1; k < 5; ++k) {
            const int i = 4 * w + k - 1, j = 2 * lane + c;
            if (i >= 1 && i < L.nz && j < W) L.e[i * W + j] = x[c][k];
        }
}

__global__ void __launch_bounds__(TAIL_THREADS) k_mg_tail(const TailRun* runs, const int* done, int sweeps,
                                                           const __grid_constant__ TailRun one) {
    extern __shared__ __align__(16) float sm[];
    __shared__ TailRun R;
    __shared__ TailLevel tl[MG_MAX_LEVELS];
    const int run = blockIdx.x;
    const int skip = done[run];
    if (threadIdx.x < sizeof(TailRun) / 4)
        reinterpret_cast<int*>(&R)[threadIdx.x] = reinterpret_cast<const int*>(gridDim.x > 1 ? runs + run : &one)[threadIdx.x];
    if (skip) return;
    __syncthreads();
    const int n = R.n;                           // levels counted from the tail's first
    if ((int)threadIdx.x < n) {
        const int l = threadIdx.x;
        const int W = R.nr[l] + 1, nodes = (R.nz[l] + 1) * W;
        TailLevel& t = tl[l];
        t.nz = R.nz[l];
        t.nr = R.nr[l];
        t.e = sm + R.node_off[l];
        t.f = t.e + nodes;
        t.r = t.f + nodes;
        t.ap = sm + R.coef_off[l];
        t.am = t.ap + W;
        t.b = t.am + W;
        t.d = t.b + W;
    }
    // inputs: the coefficients (packed as they lie in shared memory), zero
    // corrections, f of the first level; a small inverse on its way meanwhile
    if (R.inv_off >= 0)
        for (int k = threadIdx.x; k < R.inv_len / 4; k += TAIL_THREADS) {
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(sm + R.inv_off + 4 * k);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(R.inv + 4 * k) : "memory");
        }
    for (int k = threadIdx.x; k < R.ncoef; k += TAIL_THREADS) sm[k] = __ldg(&R.coef[k]);
    {
        const int nodes0 = (R.nz[0] + 1) * (R.nr[0] + 1);
        float* f0 = sm + R.node_off[0] + nodes0;
        for (int k = threadIdx.x; k < nodes0; k += TAIL_THREADS) f0[k] = R.f[k];
        for (int l = 0; l < n; ++l)
            for (int k = threadIdx.x; k < (R.nz[l] + 1) * (R.nr[l] + 1); k += TAIL_THREADS) sm[R.node_off[l] + k] = 0.0f;
    }
    __syncthreads();
    TailNode nd[2][TAIL_SLOTS];
    // down
    for (int l = 0; l + 1 < n; ++l) {
        const TailLevel F = tl[l], Cl = tl[l + 1];
        tail_nodes(F, nd);
        for (int k = 0; k < 2; ++k) {
            tail_half_sweep(F, nd[0]);
            tail_half_sweep(F, nd[1]);
        }
        const int Wf = F.nr + 1, Wc = Cl.nr + 1;
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int q = 0; q < TAIL_SLOTS; ++q) {
                const TailNode& t = nd[c][q];
                if (t.k < 0) continue;
                const int j = t.k % Wf;
                float s = (F.ap[j] + F.am[j] + 2.0f * F.b[j]) * F.e[t.k];
                s = fmaf(-t.ap, F.e[t.rt], s);
                s = fmaf(-t.am, F.e[t.lf], s);
                s = fmaf(-t.bu, F.e[t.up], s);
                s = fmaf(-t.bd, F.e[t.dn], s);
                F.r[t.k] = t.f - s;
            }
        __syncthreads();
        for (int k = threadIdx.x; k < (Cl.nz - 1) * Wc; k += TAIL_THREADS) {
            const int I = 1 + k / Wc, J = k - (I - 1) * Wc;
            float s = 0.0f;
#pragma unroll
            for (int di = -1; di <= 1; ++di) {
                const float wi = di == 0 ? 1.0f : 0.5f;
                const float* r = F.r + (2 * I + di) * Wf + 2 * J;
                if (J > 0) s = fmaf(0.5f * wi, r[-1], s);
                s = fmaf(wi, r[0], s);
                if (2 * J + 1 <= F.nr) s = fmaf(0.5f * wi, r[1], s);
            }
            Cl.f[I * Wc + J] = s;
        }
        __syncthreads();
    }
    // coarsest
    {
        const TailLevel L = tl[n - 1];
        const int W = L.nr + 1;
        const int m = (L.nz - 1) * W;
        const float* Ai = R.inv_off >= 0 ? sm + R.inv_off : R.inv;
        if (R.inv_off >= 0) {
            asm volatile("cp.async.wait_all;\n" ::: "memory");
            __syncthreads();
        }
        if (Ai) {
            // e = A^-1 f: P threads per unknown, each summing every P-th
            // term (their loads in flight together), then a shuffle sum
            const int P = m <= 64 ? 8 : (m <= 128 ? 4 : (m <= 256 ? 2 : 1));
            const int per = TAIL_THREADS / P;
            for (int u0 = 0; u0 < m; u0 += per) {        // the same trip count in every thread
                const int u = u0 + (int)threadIdx.x / P, part = (int)threadIdx.x % P;
                float acc = 0.0f;
                if (u < m) {
#pragma unroll 8
                    for (int v = part; v < m; v += P) acc += Ai[(size_t)v * m + u] * L.f[W + v];
                }
                for (int o = P >> 1; o > 0; o >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, o, P);
                if (part == 0 && u < m) L.e[W + u] = acc;
            }
            __syncthreads();
        } else if (L.nz <= GS_DIM && W <= GS_DIM) {
            const int warps = (L.nz + 3) / 4;
            if ((int)threadIdx.x < 32 * warps) tail_sweeps_rows(L, sweeps, warps);
            __syncthreads();
        } else {
            tail_nodes(L, nd);
            for (int it = 0; it < sweeps; ++it) {
                tail_half_sweep(L, nd[0]);
                tail_half_sweep(L, nd[1]);
            }
        }
    }
    // up
    for (int l = n - 2; l >= 0; --l) {
        const TailLevel F = tl[l], Cl = tl[l + 1];
        const int Wf = F.nr + 1, Wc = Cl.nr + 1;
        tail_nodes(F, nd);
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int q = 0; q < TAIL_SLOTS; ++q) {
                const int k = nd[c][q].k;
                if (k < 0) continue;
                const int i = k / Wf, j = k - i * Wf;
                const int I0 = i >> 1, J0 = j >> 1;
                const int I1 = (i & 1) ? I0 + 1 : I0, J1 = (j & 1) ? J0 + 1 : J0;
                const float s =
                    ((Cl.e[I0 * Wc + J0] + Cl.e[I1 * Wc + J0]) + Cl.e[I0 * Wc + J1]) + Cl.e[I1 * Wc + J1];
                F.e[k] = fmaf(0.25f, s, F.e[k]);
            }
        __syncthreads();
        for (int k = 0; k < 2; ++k) {
            tail_half_sweep(F, nd[1]);
            tail_half_sweep(F, nd[0]);
        }
    }
    // output
    const TailLevel t = tl[0];
    const int W = t.nr + 1;
    if (R.phi) {
        double* phi = R.phi;
        for (int q = threadIdx.x; q < (t.nz - 1) * W; q += TAIL_THREADS) phi[W + q] += (double)t.e[W + q];
    } else {
        float* e = R.e;
        for (int k = threadIdx.x; k < (t.nz + 1) * W; k += TAIL_THREADS) e[k] = t.e[k];
    }
}

// E = -grad(phi): central inside, one-sided at the electrodes, E_r = 0 on the
// axis and at r = R; and the end of the solve's bookkeeping
__global__ void k_efield(const MGTop* top, const RunInfo* runs, float2* E, const int* done, DevState* st,
                         RunState* rs) {
    const int run = blockIdx.y;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (done[run] == 2) atomicOr(&st->error, ERR_NONFINITE);
        const double rel = rs[run].relres;
        if (!(rel <= rs[run].relres_max)) rs[run].relres_max = rel;   // NaN propagates
    }
    const MGTop T = top[run];
    const int nz = T.nz, nr = T.nr;
    const int W = nr + 1;
    const int n = (nz + 1) * W;
    const double* p = T.phi;
    float2* out = E + runs[run].node_base;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int i = k / W, j = k - i * W;
        double ez, er;
        if (i == 0) ez = -(p[k + W] - p[k]) * T.idz;
        else if (i == nz) ez = -(p[k] - p[k - W]) * T.idz;
        else ez = -(p[k + W] - p[k - W]) * T.i2dz;
        if (j == 0 || j == nr) er = 0.0;
        else er = -(p[k + 1] - p[k - 1]) * T.i2dr;
        out[k] = make_float2((float)ez, (float)er);
    }
}

// ------------------------------------------------------------------
// host
// ------------------------------------------------------------------
static int blocks_for(const FieldSolver& fs, int n) {
    int b = (n + fs.threads - 1) / fs.threads;
    return b < 1 ? 1 : (b > fs.max_blocks ? fs.max_blocks : b);
}

// Inverse of the coarsest operator by Gauss-Jordan elimination with partial
// pivoting; unknown u = (i - 1) (nr + 1) + j for interior rows i and radial
// nodes j, the rows of the smoother's equation.  Stored transposed.
static bool invert_coarse(int nz, int nr, const std::vector<double>& ap, const std::vector<double>& am,
                          const std::vector<double>& bb, std::vector<double>& out) {
    const int W = nr + 1, m = (nz - 1) * W;
    std::vector<double> A((size_t)m * m, 0.0), X((size_t)m * m, 0.0);
    for (int u = 0; u < m; ++u) {
        const int i = 1 + u / W, j = u % W;
        A[(size_t)u * m + u] = ap[j] + am[j] + 2.0 * bb[j];
        if (j < nr) A[(size_t)u * m + u + 1] = -ap[j];
        if (j > 0) A[(size_t)u * m + u - 1] = -am[j];
        if (i + 1 < nz) A[(size_t)u * m + u + W] = -bb[j];
        if (i - 1 > 0) A[(size_t)u * m + u - W] = -bb[j];
        X[(size_t)u * m + u] = 1.0;
    }
    for (int c = 0; c < m; ++c) {
        int p = c;
        for (int r = c + 1; r < m; ++r)
            if (std::fabs(A[(size_t)r * m + c]) > std::fabs(A[(size_t)p * m + c])) p = r;
        if (!(std::fabs(A[(size_t)p * m + c]) > 0.0)) return false;
        if (p != c)
            for (int k = 0; k < m; ++k) {
                std::swap(A[(size_t)p * m + k], A[(size_t)c * m + k]);
                std::swap(X[(size_t)p * m + k], X[(size_t)c * m + k]);
            }
        const double d = A[(size_t)c * m + c];
        for (int k = 0; k < m; ++k) {
            A[(size_t)c * m + k] /= d;
            X[(size_t)c * m + k] /= d;
        }
        for (int r = 0; r < m; ++r) {
            if (r == c) continue;
            const double f = A[(size_t)r * m + c];
            if (f == 0.0) continue;
            for (int k = 0; k < m; ++k) {
                A[(size_t)r * m + k] -= f * A[(size_t)c * m + k];
                X[(size_t)r * m + k] -= f * X[(size_t)c * m + k];
            }
        }
    }
    out.assign((size_t)m * m, 0.0);
    for (int u = 0; u < m; ++u)
        for (int v = 0; v < m; ++v) out[(size_t)v * m + u] = X[(size_t)u * m + v];
    return true;
}

// coefficients of one level (cell sizes dz, dr, nr cells radially)
static void level_coeffs(int nr, double dz, double dr, std::vector<double>& ap, std::vector<double>& am,
                         std::vector<double>& bb) {
    ap.assign(nr + 1, 0.0);
    am.assign(nr + 1, 0.0);
    bb.assign(nr + 1, 0.0);
    const double Rr = nr * dr;
    for (int j = 0; j <= nr; ++j) {
        const double rp = (j + 0.5) * dr, rm = (j - 0.5) * dr;
        ap[j] = j < nr ? 2.0 * PI_ * rp * dz / dr : 0.0;
        am[j] = j > 0 ? 2.0 * PI_ * rm * dz / dr : 0.0;
        double A;
        if (j == 0) A = PI_ * (0.5 * dr) * (0.5 * dr);
        else if (j == nr) A = PI_ * (Rr * Rr - (Rr - 0.5 * dr) * (Rr - 0.5 * dr));
        else A = 2.0 * PI_ * j * dr * dr;
        bb[j] = A / dz;
    }
}

template <typename T>
static void upload(T* dst, const std::vector<T>& v, cudaStream_t s) {
    cudaMemcpyAsync(dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, s);
}

static std::vector<float> to_float(const std::vector<double>& v) { return std::vector<float>(v.begin(), v.end()); }

int field_init(FieldSolver& fs, const std::vector<pd_config>& cfgs, const std::vector<uint32_t>& node_base,
               double* phi, void* ws, size_t bytes, cudaStream_t s) {
    const int R = (int)cfgs.size();
    {
        std::vector<int> nz(R), nr(R);
        for (int r = 0; r < R; ++r) {
            nz[r] = cfgs[r].nz;
            nr[r] = cfgs[r].nr;
        }
        if (field_workspace_bytes(nz, nr) > bytes) return 1;   // checked before anything is written
    }
    char* w = (char*)ws;
    size_t o = 0;
    auto take = [&](size_t sz) {
        char* p = w + o;
        o += al(sz);
        return p;
    };
    // every array starts at zero (the electrode rows of the corrections stay zero)
    if (cudaMemsetAsync(ws, 0, bytes, s) != cudaSuccess) return 1;
    fs.nruns = R;
    fs.host_lev.assign((size_t)R * MG_MAX_LEVELS, MGLevel{});
    fs.host_top.assign(R, MGTop{});
    fs.max_tail = 0;
    fs.tail_smem = 0;
    fs.tail_lev.assign(R, 0);
    fs.max_nodes0 = 0;
    fs.max_cycles = cfgs[0].poisson_max_cycles > 0 ? cfgs[0].poisson_max_cycles : 60;
    std::vector<double> tol(R);
    std::vector<TailRun> tails(R, TailRun{});
    for (int r = 0; r < R; ++r) {
        const pd_config& c = cfgs[r];
        int a[MG_MAX_LEVELS], b[MG_MAX_LEVELS], n;
        level_dims(c.nz, c.nr, a, b, n);
        fs.tail_lev[r] = tail_level(a, b, n);
        fs.max_tail = std::max(fs.max_tail, fs.tail_lev[r]);
        fs.max_nodes0 = std::max(fs.max_nodes0, (c.nz + 1) * (c.nr + 1));
        tol[r] = c.poisson_tol;
        // level 0 in double
        MGTop& T = fs.host_top[r];
        const size_t W0 = (size_t)c.nr + 1, nodes0 = ((size_t)c.nz + 1) * W0;
        T.nz = c.nz;
        T.nr = c.nr;
        T.phi = phi + node_base[r];
        T.bf = (double*)take(nodes0 * 8);
        T.ap = (double*)take(W0 * 8);
        T.am = (double*)take(W0 * 8);
        T.b = (double*)take(W0 * 8);
        T.dg = (double*)take(W0 * 8);
        T.cr = (double*)take(W0 * 8);
        T.iv = (double*)take(W0 * 8);
        T.idz = 1.0 / c.dz;
        T.i2dz = 1.0 / (2.0 * c.dz);
        T.i2dr = 1.0 / (2.0 * c.dr);
        std::vector<double> ap, am, bb;
        level_coeffs(c.nr, c.dz, c.dr, ap, am, bb);
        std::vector<double> cr(W0), iv(W0);
        const double qw = QE_ * c.weight / 4294967296.0;
        for (int j = 0; j <= c.nr; ++j) {
            double verb;     // Verboncoeur volume of an interior node
            if (j == 0) verb = PI_ * c.dz * c.dr * c.dr / 3.0;
            else if (j == c.nr) verb = 2.0 * PI_ * c.dz * c.dr * c.dr * ((double)c.nr / 2.0 - 1.0 / 6.0);
            else verb = 2.0 * PI_ * c.dz * c.dr * c.dr * (double)j;
            const double vfv = bb[j] * c.dz * c.dz;   // finite volume: radial extent area x dz
            iv[j] = 1.0 / verb;
            cr[j] = qw * vfv / (verb * EPS0_);        // b = (charge / verb) vfv / eps0
        }
        upload(T.ap, ap, s);
        upload(T.am, am, s);
        upload(T.b, bb, s);
        std::vector<double> dg(W0);
        for (size_t j = 0; j < W0; ++j) dg[j] = ap[j] + am[j] + 2.0 * bb[j];
        upload(T.dg, dg, s);
        upload(T.cr, cr, s);
        upload(T.iv, iv, s);
        cudaStreamSynchronize(s);          // the host vectors above go out of scope
        // correction levels in float
        std::vector<float> coef;
        for (int l = 0; l < n; ++l) {
            MGLevel& L = fs.host_lev[(size_t)r * MG_MAX_LEVELS + l];
            L.nz = a[l];
            L.nr = b[l];
            const double dz = c.dz * (double)(1 << l), dr = c.dr * (double)(1 << l);
            const size_t W = (size_t)L.nr + 1, nodes = ((size_t)L.nz + 1) * W;
            L.e = (float*)take(nodes * 4);
            L.e2 = (float*)take(nodes * 4);
            L.f = (float*)take(nodes * 4);
            L.ap = (float*)take(W * 4);
            L.am = (float*)take(W * 4);
            L.b = (float*)take(W * 4);
            L.dinv = (float*)take(W * 4);
            std::vector<double> lap, lam, lbb;
            level_coeffs(L.nr, dz, dr, lap, lam, lbb);
            std::vector<double> dinv(W);
            for (size_t j = 0; j < W; ++j) dinv[j] = 1.0 / (lap[j] + lam[j] + 2.0 * lbb[j]);
            const std::vector<float> fap = to_float(lap), fam = to_float(lam), fbb = to_float(lbb),
                                     fdi = to_float(dinv);
            upload(L.ap, fap, s);
            upload(L.am, fam, s);
            upload(L.b, fbb, s);
            upload(L.dinv, fdi, s);
            std::vector<float> fai;
            if (l == n - 1 && coarse_unknowns(a, b, n) <= MG_DIRECT_MAX) {
                const int m = coarse_unknowns(a, b, n);
                std::vector<double> Ai;
                if (!invert_coarse(L.nz, L.nr, lap, lam, lbb, Ai)) return 1;
                float* inv = (float*)take((size_t)m * m * 4 + 16);
                fai = to_float(Ai);
                upload(inv, fai, s);
                tails[r].inv = inv;
                if (m <= INV_SMEM) tails[r].inv_len = (m * m + 3) / 4 * 4;
            }
            cudaStreamSynchronize(s);      // the host vectors above go out of scope
            if (l >= fs.tail_lev[r])
                for (const std::vector<float>* v : {&fap, &fam, &fbb, &fdi}) coef.insert(coef.end(), v->begin(), v->end());
        }
        // k_mg_tail's table
        TailRun& tr = tails[r];
        const int t0 = fs.tail_lev[r];
        int o_coef = 0, o_node = (int)coef.size();
        tr.n = n - t0;
        tr.ncoef = o_node;
        for (int l = t0; l < n; ++l) {
            tr.nz[l - t0] = a[l];
            tr.nr[l - t0] = b[l];
            tr.coef_off[l - t0] = o_coef;
            tr.node_off[l - t0] = o_node;
            o_coef += 4 * (b[l] + 1);
            o_node += 3 * (a[l] + 1) * (b[l] + 1);
        }
        tr.inv_off = -1;
        if (tr.inv_len) {
            tr.inv_off = (o_node + 3) / 4 * 4;
            o_node = tr.inv_off + tr.inv_len;
        }
        fs.tail_smem = std::max(fs.tail_smem, (size_t)o_node * sizeof(float));
        float* dcoef = (float*)take(coef.size() * 4);
        upload(dcoef, coef, s);
        cudaStreamSynchronize(s);
        tr.coef = dcoef;
        tr.f = fs.host_lev[(size_t)r * MG_MAX_LEVELS + t0].f;
        tr.e = fs.host_lev[(size_t)r * MG_MAX_LEVELS + t0].e;
        tr.phi = t0 == 0 ? T.phi : nullptr;
    }
    fs.lev = (MGLevel*)take((size_t)R * MG_MAX_LEVELS * sizeof(MGLevel));
    fs.top = (MGTop*)take((size_t)R * sizeof(MGTop));
    fs.done = (int*)take((size_t)R * 4);
    fs.ticket = (unsigned int*)take((size_t)R * 4);
    fs.red_base = (int*)take((size_t)R * 4);
    std::vector<int> red_base(R);
    int nred = 0;
    for (int r = 0; r < R; ++r) {
        red_base[r] = nred;
        nred += red_blocks(cfgs[r].nz, cfgs[r].nr);
    }
    fs.red = (double*)take((size_t)nred * 2 * 8);
    fs.bnorm = (double*)take((size_t)R * 8);
    fs.tol = (double*)take((size_t)R * 8);
    fs.tails = (TailRun*)take((size_t)R * sizeof(TailRun));
    // work lists, level by level: the levels above each run's tail
    std::vector<int2> tasks;
    for (int l = 0; l < MG_MAX_LEVELS; ++l) {
        // short windows where long ones would leave most SMs idle: a tile of
        // K = 20 rows is through in two thirds of the time of one of 32, but
        // spends 60 % of its rows on the rings instead of 38 %; the line is four
        // tiles, one block, an SM
        int large = 0;
        for (int r = 0; r < R; ++r)
            if (l < fs.tail_lev[r]) large += tiles_of(fs.host_lev[(size_t)r * MG_MAX_LEVELS + l].nz,
                                                      fs.host_lev[(size_t)r * MG_MAX_LEVELS + l].nr, K_LARGE, PRE_H);
        fs.rows[l] = large > SMALL_TILES ? K_LARGE : K_SMALL;
        for (int post = 0; post < 2; ++post) {
            fs.tile_off[post][l] = (int)tasks.size();
            for (int r = 0; r < R; ++r)
                if (l < fs.tail_lev[r]) {
                    const MGLevel& L = fs.host_lev[(size_t)r * MG_MAX_LEVELS + l];
                    const int cnt = tiles_of(L.nz, L.nr, fs.rows[l], post ? POST_H : PRE_H);
                    for (int q = 0; q < cnt; ++q) tasks.push_back(make_int2(r, q));
                }
            fs.tile_len[post][l] = (int)tasks.size() - fs.tile_off[post][l];
        }
    }
    fs.red_off = (int)tasks.size();
    for (int r = 0; r < R; ++r)
        for (int u = 0; u < red_units(cfgs[r].nz, cfgs[r].nr); u += RED_WARPS) tasks.push_back(make_int2(r, u));
    fs.red_len = (int)tasks.size() - fs.red_off;
    // The limit is the kernel's, shared by every solver of the process: always the
    // same value, so that no solver lowers it under another's launches.
    if (fs.tail_smem > TAIL_SMEM_MAX) return 1;
    if (cudaFuncSetAttribute(k_mg_tail, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TAIL_SMEM_MAX) != cudaSuccess)
        return 1;
    fs.tasks = (int2*)take(tasks.size() * sizeof(int2) + 8);
    if (o > bytes) return 1;
    upload(fs.tasks, tasks, s);
    upload(fs.lev, fs.host_lev, s);
    upload(fs.top, fs.host_top, s);
    upload(fs.tol, tol, s);
    upload(fs.tails, tails, s);
    fs.host_tail = tails[0];
    upload(fs.red_base, red_base, s);
    if (!fs.host_done && cudaMallocHost(&fs.host_done, (size_t)R * 4) != cudaSuccess) return 1;
    return cudaStreamSynchronize(s) == cudaSuccess ? 0 : 1;
}

void field_free(FieldSolver& fs) {
    if (fs.host_done) cudaFreeHost(fs.host_done);
    fs.host_done = nullptr;
}

// A single run's levels go to the kernels by value, and its tiles are numbered as
// they lie (no task list): two dependent reads fewer before the first load of the
// data, and the convergence flag is read beside it.  512 x 512 cells, a launch under
// ncu: k_down 5.2 -> 4.1 us, k_up 6.5 -> 5.5, residual 15.1 -> 14.5.
//
// one correction cycle of every run that has not converged (the right-hand
// side is level 0's f, set with the residual norms); returns the kernels
// launched
static int vcycle(FieldSolver& fs, cudaStream_t s) {
    const int R = fs.nruns, th = TILE_WARPS * 32;
    int nk = 1;
    // down to each run's tail: pre-smooth, residual and restriction
    for (int l = 0; l < fs.max_tail; ++l) {
        const int n = fs.tile_len[0][l], g = (n + TILE_WARPS - 1) / TILE_WARPS;
        const int2* t = R > 1 ? fs.tasks + fs.tile_off[0][l] : nullptr;
        const MGLevel& L = fs.host_lev[l];
        if (!n) continue;
        if (fs.rows[l] == K_SMALL) k_down<K_SMALL><<<g, th, 0, s>>>(fs.lev, fs.done, l, t, n, L);
        else k_down<K_LARGE><<<g, th, 0, s>>>(fs.lev, fs.done, l, t, n, L);
        ++nk;
    }
    // the tail levels of every run, one block each
    k_mg_tail<<<R, TAIL_THREADS, fs.tail_smem, s>>>(fs.tails, fs.done, 200, fs.host_tail);
    // up: prolongation and post-smoothing in one launch per level; level 0's adds the correction to phi
    for (int l = fs.max_tail - 1; l >= 0; --l) {
        const int n = fs.tile_len[1][l], g = (n + TILE_WARPS - 1) / TILE_WARPS;
        const int2* t = R > 1 ? fs.tasks + fs.tile_off[1][l] : nullptr;
        const MGLevel &L = fs.host_lev[l], &C = fs.host_lev[l + 1];
        double* phi = fs.host_top[0].phi;
        if (!n) continue;
        const bool small = fs.rows[l] == K_SMALL;
        if (l == 0 && small) k_up<K_SMALL, true><<<g, th, 0, s>>>(fs.lev, fs.top, fs.done, l, t, n, L, C, phi);
        else if (l == 0) k_up<K_LARGE, true><<<g, th, 0, s>>>(fs.lev, fs.top, fs.done, l, t, n, L, C, phi);
        else if (small) k_up<K_SMALL, false><<<g, th, 0, s>>>(fs.lev, fs.top, fs.done, l, t, n, L, C, phi);
        else k_up<K_LARGE, false><<<g, th, 0, s>>>(fs.lev, fs.top, fs.done, l, t, n, L, C, phi);
        ++nk;
    }
    return nk;
}

static void norms(FieldSolver& fs, RunState* rs, int cycle, cudaStream_t s) {
    k_residual_norms<<<fs.red_len, 32 * RED_WARPS, 0, s>>>(
        fs.top, fs.lev, fs.nruns > 1 ? fs.tasks + fs.red_off : nullptr, fs.red_base, fs.red, fs.ticket, fs.bnorm, fs.done,
        fs.tol, rs, cycle, fs.host_top[0], fs.host_lev[0].f);
}

cudaError_t field_solve(FieldSolver& fs, RunState* rs, int host_check, int cycles, cudaStream_t s, int* kernels) {
    const int R = fs.nruns;
    norms(fs, rs, 0, s);
    if (kernels) *kernels += 1;
    if (host_check) {
        for (int cyc = 1; cyc <= fs.max_cycles; ++cyc) {
            cudaError_t e = cudaMemcpyAsync(fs.host_done, fs.done, (size_t)R * 4, cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) return e;
            bool all = true;
            for (int r = 0; r < R; ++r) all = all && fs.host_done[r] != 0;
            if (all) break;
            const int nk = vcycle(fs, s);
            norms(fs, rs, cyc, s);
            if (kernels) *kernels += nk + 1;
        }
    } else {
        for (int cyc = 1; cyc <= cycles; ++cyc) {
            const int nk = vcycle(fs, s);
            norms(fs, rs, cyc, s);
            if (kernels) *kernels += nk + 1;
        }
    }
    return cudaGetLastError();
}

// E for every run (separate so the caller can time it)
void field_efield(FieldSolver& fs, const double* phi, const RunInfo* runs, float2* E, DevState* st, RunState* rs,
                  cudaStream_t s) {
    (void)phi;
    const dim3 g(blocks_for(fs, fs.max_nodes0), fs.nruns);
    k_efield<<<g, fs.threads, 0, s>>>(fs.top, runs, E, fs.done, st, rs);
}

// ------------------------------------------------------------------
// warm start
// ------------------------------------------------------------------
// The start of a solve: the right-hand side b (double) and the electrode rows
// of phi (blockIdx.y = run), and the history shift rho_prev2 := rho_prev,
// rho_prev := rho_last, phi_prev2 := phi_prev, phi_prev := phi, V_prev2 :=
// V_prev, V_prev := V_last; then rho_last := current density, V_last := V.
__global__ void k_begin(const long long* rho_e, const long long* rho_h, const MGTop* top, const RunInfo* runs,
                        const RunState* rs, WarmHistory h, int extrapolate) {
    const int run = blockIdx.y;
    const MGTop& T = top[run];
    const RunInfo& RI = runs[run];
    const double qw = QE_ * RI.weight / 4294967296.0, V = rs[run].V;
    const int nz = T.nz, W = T.nr + 1, n = (nz + 1) * W;
    double *phi = T.phi, *bf = T.bf;
    const double *cr = T.cr, *iv = T.iv, *bz = T.b;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int i = k / W, j = k - i * W;
        const bool rim = i == 0 || i == nz;
        const uint32_t g = RI.node_base + (uint32_t)k;
        const double q = (double)(rho_e[g] + rho_h[g]);
        h.rho_prev2[g] = h.rho_prev[g];
        h.rho_prev[g] = h.rho_last[g];
        const double p = phi[k], pp = h.phi_prev[g];
        if (rim) phi[k] = i == 0 ? 0.0 : V;
        else if (extrapolate) phi[k] = 2.0 * p - pp;
        double v = 0.0;
        if (!rim) {
            v = q * cr[j];
            if (i == nz - 1) v += bz[j] * V;
        }
        bf[k] = v;
        h.phi_prev2[g] = pp;
        h.phi_prev[g] = p;
        h.rho_last[g] = qw * q * (iv[j] * (rim ? 2.0 : 1.0));       // half volume on the electrode rows
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        h.V_prev2[run] = h.V_prev[run];
        h.V_prev[run] = h.V_last[run];
        h.V_last[run] = V;
    }
}

// The references of a form: d = rho_last - c1 rho1 - c2 rho2 and base =
// c1 phi1 + c2 phi2 + (V - c1 V1 - c2 V2) z / L (absent terms: 0)
struct WarmRef {
    const double *rho1, *rho2, *phi1, *phi2, *V1, *V2;
    double c1, c2;
};

WarmRef warm_ref(const WarmHistory& h, int form) {
    WarmRef r{nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0.0, 0.0};
    if (form == WARM_DELTA) {
        r.rho1 = h.rho_prev;
        r.phi1 = h.phi_prev;
        r.V1 = h.V_prev;
        r.c1 = 1.0;
    } else if (form == WARM_EXTRAP) {
        r.rho1 = h.rho_prev;
        r.phi1 = h.phi_prev;
        r.V1 = h.V_prev;
        r.c1 = 2.0;
        r.rho2 = h.rho_prev2;
        r.phi2 = h.phi_prev2;
        r.V2 = h.V_prev2;
        r.c2 = -1.0;
    }
    return r;
}

__device__ __forceinline__ double warm_d(const double* rho_last, const WarmRef& R, uint32_t g) {
    double d = rho_last[g];
    if (R.rho1) d -= R.c1 * R.rho1[g];
    if (R.rho2) d -= R.c2 * R.rho2[g];
    return d;
}

// rmax[run] = max |d|
__global__ void k_warm_rmax(const double* rho_last, WarmRef R, const RunInfo* runs, unsigned long long* rmax_bits) {
    const int run = blockIdx.y;
    const RunInfo& RI = runs[run];
    const int n = (RI.nz + 1) * (RI.nr + 1);
    double m = 0.0;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x)
        m = fmax(m, fabs(warm_d(rho_last, R, RI.node_base + (uint32_t)k)));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xFFFFFFFFu, m, o));
    // non-negative doubles order like their bit patterns
    if ((threadIdx.x & 31) == 0 && m > 0.0) atomicMax(&rmax_bits[run], (unsigned long long)__double_as_longlong(m));
}

__global__ void k_warm_x(const double* rho_last, WarmRef R, const RunInfo* runs, const double* rmax, float* x) {
    const int run = blockIdx.y;
    const RunInfo& RI = runs[run];
    const int n = (RI.nz + 1) * (RI.nr + 1);
    const double rm = rmax[run];
    const double irm = rm > 0.0 ? 1.0 / rm : 0.0;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const uint32_t g = RI.node_base + (uint32_t)k;
        x[g] = (float)(warm_d(rho_last, R, g) * irm);
    }
}

// the potential the prediction is added to
__device__ __forceinline__ double warm_base(const WarmRef& R, int run, double V, uint32_t g, int i, double inz) {
    double b = 0.0, Vr = 0.0;
    if (R.phi1) {
        b += R.c1 * R.phi1[g];
        Vr += R.c1 * R.V1[run];
    }
    if (R.phi2) {
        b += R.c2 * R.phi2[g];
        Vr += R.c2 * R.V2[run];
    }
    return b + (V - Vr) * ((double)i * inz);
}

__global__ void k_warm_apply(const float* y, const MGTop* top, const RunInfo* runs, const RunState* rs,
                             const double* rmax, WarmRef R, double* phi) {
    const int run = blockIdx.y;
    const RunInfo& RI = runs[run];
    const MGTop T = top[run];
    const int W = RI.nr + 1, n = (RI.nz - 1) * W;
    const double V = rs[run].V, inz = 1.0 / (double)RI.nz;
    const double dz = 1.0 / T.idz;
    const double sc = y ? rmax[run] * dz * dz / EPS0_ : 0.0;
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        const int i = 1 + q / W;
        const uint32_t g = RI.node_base + (uint32_t)(W + q);
        const double base = warm_base(R, run, V, g, i, inz);
        phi[g] = y ? base + (double)y[g] * sc : base;
    }
}

__global__ void k_warm_targets(const double* phi, const MGTop* top, const RunInfo* runs, const double* V_last,
                               const double* rmax, WarmRef R, float* t) {
    const int run = blockIdx.y;
    const RunInfo& RI = runs[run];
    const MGTop T = top[run];
    const int W = RI.nr + 1, n = (RI.nz + 1) * W;
    const double V = V_last[run], rm = rmax[run], inz = 1.0 / (double)RI.nz;
    const double dz = 1.0 / T.idz;
    const double sc = rm > 0.0 ? EPS0_ / (rm * dz * dz) : 0.0;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int i = k / W;
        const uint32_t g = RI.node_base + (uint32_t)k;
        t[g] = (float)((phi[g] - warm_base(R, run, V, g, i, inz)) * sc);
    }
}

void field_begin(FieldSolver& fs, const long long* rho_e, const long long* rho_h, const RunInfo* runs,
                 const RunState* rs, const WarmHistory& h, bool extrapolate, cudaStream_t s) {
    const dim3 g(blocks_for(fs, fs.max_nodes0), fs.nruns);
    k_begin<<<g, fs.threads, 0, s>>>(rho_e, rho_h, fs.top, runs, rs, h, extrapolate ? 1 : 0);
}

void warm_inputs(FieldSolver& fs, const WarmHistory& h, int form, const RunInfo* runs, double* rmax, float* x,
                 cudaStream_t s) {
    const dim3 g(blocks_for(fs, fs.max_nodes0), fs.nruns);
    const WarmRef R = warm_ref(h, form);
    cudaMemsetAsync(rmax, 0, (size_t)fs.nruns * 8, s);
    k_warm_rmax<<<g, fs.threads, 0, s>>>(h.rho_last, R, runs, (unsigned long long*)rmax);
    k_warm_x<<<g, fs.threads, 0, s>>>(h.rho_last, R, runs, rmax, x);
}

void warm_apply(FieldSolver& fs, const float* y, const WarmHistory& h, int form, const RunInfo* runs,
                const RunState* rs, const double* rmax, double* phi, cudaStream_t s) {
    const dim3 g(blocks_for(fs, fs.max_nodes0), fs.nruns);
    k_warm_apply<<<g, fs.threads, 0, s>>>(y, fs.top, runs, rs, rmax, warm_ref(h, form), phi);
}

void warm_targets(FieldSolver& fs, const double* phi, const WarmHistory& h, int form, const RunInfo* runs,
                  const double* rmax, float* t, cudaStream_t s) {
    const dim3 g(blocks_for(fs, fs.max_nodes0), fs.nruns);
    k_warm_targets<<<g, fs.threads, 0, s>>>(phi, fs.top, runs, h.V_last, rmax, warm_ref(h, form), t);
}

}  // namespace pd
