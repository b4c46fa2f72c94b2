// pd_collide.cu -- DSMC electron-impact collisions and cathode injection.
//
// Collisions (Sec. 2.1 Eq. (4)-(7), Sec. 2.2 Eq. (11)-(20)) in no-time-counter
// form, per cell and pair class k in {(e, Cu), (e, Cu+)}:
//   k_ncand    N_cand = floor(N_e N_t c_k(r) + R), c_k = W (sigma g)_max dt_coll / V_cell,
//              one thread per cell; cells with candidates go to an active list.
//              Lists of more than RANK_WARP_MAX ids that active cells use
//              are queued for k_rank_tables.
//   k_rank_tables  rank tables of the queued lists, one block per list.
//   k_collide  one warp per active cell, or a block per cell of BIG_CELL
//              candidates or more.  Candidate m draws from the stream
//              (cell, step, k<<28 | m): the electron and target ranks (in
//              ascending-id order inside the cell), the acceptance number and
//              the channel number.  A batch (a candidate a thread) is applied in
//              rounds: in each, the candidates whose earlier sharers of a particle
//              are through, side by side.  Spawned electrons go to the slots
//              reserved for the cell at n_alive + 2 * (candidates of the
//              cells before it); unused reserved slots are marked dead.
//   k_coulomb  one warp per batch of cells: the Coulomb pairs (see there).
//   k_finalize slot / id bookkeeping and the RC circuit update.
// Compiled with -fmad=false (decision arithmetic is rounded op by op).
#include <algorithm>

#include "pd_internal.cuh"
#include "pd_kernels.h"

namespace pd {

constexpr unsigned FULL = 0xFFFFFFFFu;

struct V3 {
    float x, y, z;
};

// isotropic unit vector, Marsaglia (1972)
template <typename S>
__device__ __forceinline__ V3 iso_dir(S& st, uint32_t& fb) {
#pragma unroll 1
    for (int a = 0; a < 64; ++a) {
        const float u1 = 2.0f * st.u01() - 1.0f;
        const float u2 = 2.0f * st.u01() - 1.0f;
        const float s = u1 * u1 + u2 * u2;
        if (s < 1.0f) {
            const float q = 2.0f * sqrtf(1.0f - s);
            return V3{u1 * q, u2 * q, 1.0f - 2.0f * s};
        }
    }
    ++fb;
    return V3{0.0f, 0.0f, 1.0f};
}

// uniform azimuth (cos, sin) from a point of the unit disc
template <typename S>
__device__ __forceinline__ void azimuth(S& st, float& c, float& s, uint32_t& fb) {
#pragma unroll 1
    for (int a = 0; a < 64; ++a) {
        const float u1 = 2.0f * st.u01() - 1.0f;
        const float u2 = 2.0f * st.u01() - 1.0f;
        const float q = u1 * u1 + u2 * u2;
        if (q < 1.0f && q > 0.0f) {
            const float r = sqrtf(q);
            c = u1 / r;
            s = u2 / r;
            return;
        }
    }
    ++fb;
    c = 1.0f;
    s = 0.0f;
}

// Eq. (6): |u'|^2 = |u|^2 - 2 E_th / m_r (kth); Eq. (7) isotropic direction;
// Eq. (5): v1 += (u' - u) m_r/m1, v2 -= (u' - u) m_r/m2.
template <typename S>
__device__ __forceinline__ bool binary_scatter(S& st, V3& v1, V3& v2, float kth, float a1, float a2, uint32_t& fb) {
    const V3 u{v1.x - v2.x, v1.y - v2.y, v1.z - v2.z};
    const float g2 = (u.x * u.x + u.y * u.y) + u.z * u.z;
    const float up2 = g2 - kth;
    if (up2 < 0.0f) return false;
    const float gp = sqrtf(up2);
    const V3 n = iso_dir(st, fb);
    const V3 du{gp * n.x - u.x, gp * n.y - u.y, gp * n.z - u.z};
    v1.x = v1.x + du.x * a1;
    v1.y = v1.y + du.y * a1;
    v1.z = v1.z + du.z * a1;
    v2.x = v2.x - du.x * a2;
    v2.y = v2.y - du.y * a2;
    v2.z = v2.z - du.z * a2;
    return true;
}

// Eq. (15)-(20): v5 = cos(chi) |v| R^T(theta, phi) (sin chi cos psi,
// sin chi sin psi, cos chi); v6 = v - v5; theta, phi from the components of v.
template <typename S>
__device__ __forceinline__ void rectangle_split(S& st, const V3& v, V3& v5, V3& v6, int mode, uint32_t& fb) {
    float cchi = st.u01();
    if (mode == 1) cchi = sqrtf(cchi);
    const float schi = sqrtf(1.0f - cchi * cchi);
    float cpsi, spsi;
    azimuth(st, cpsi, spsi, fb);
    const float vperp2 = v.x * v.x + v.y * v.y;
    const float vmag2 = vperp2 + v.z * v.z;
    const float vmag = sqrtf(vmag2), vperp = sqrtf(vperp2);
    V3 w5{0.0f, 0.0f, 0.0f};
    if (vmag > 0.0f) {
        const float ct = v.z / vmag, sth = vperp / vmag;
        float cp = 1.0f, sp = 0.0f;
        if (vperp > 0.0f) {
            cp = v.x / vperp;
            sp = v.y / vperp;
        }
        const float a = cchi * vmag;
        const float w1 = a * (schi * cpsi), w2 = a * (schi * spsi), w3 = a * cchi;
        w5.x = (w1 * (ct * cp) - w2 * sp) + w3 * (sth * cp);
        w5.y = (w1 * (ct * sp) + w2 * cp) + w3 * (sth * sp);
        w5.z = w3 * ct - w1 * sth;
    }
    v5 = w5;
    v6 = V3{v.x - w5.x, v.y - w5.y, v.z - w5.z};
}

// single-particle fixed-point CIC deposit of zq at (local cell, pz, pr) of run RI
__device__ __noinline__ void deposit1(long long* rho, const RunInfo& RI, int geom, uint32_t lcell, float pz, float pr, int zq) {
    const int iz = (int)(lcell / (uint32_t)RI.nr);
    const int ir = (int)(lcell - (uint32_t)iz * (uint32_t)RI.nr);
    const uint32_t wz = __float2uint_rn(pz * 65536.0f);
    const uint32_t wr = __float2uint_rn(pr * 65536.0f);
    const long long az = 65536 - (long long)wz, ar = 65536 - (long long)wr;
    atomicAdd((unsigned long long*)&rho[node_of(RI, geom, iz, ir)], (unsigned long long)(zq * az * ar));
    atomicAdd((unsigned long long*)&rho[node_of(RI, geom, iz + 1, ir)], (unsigned long long)(zq * (long long)wz * ar));
    atomicAdd((unsigned long long*)&rho[node_of(RI, geom, iz, ir + 1)], (unsigned long long)(zq * az * (long long)wr));
    atomicAdd((unsigned long long*)&rho[node_of(RI, geom, iz + 1, ir + 1)],
              (unsigned long long)(zq * (long long)wz * (long long)wr));
}

// Ranks inside a cell.  The candidate draws give ranks in ascending-id order;
// the sorted slots hold a cell's particles in an order that depends on the
// scatter's atomics, so each list the candidates use is mapped rank ->
// position by one of:
//   * ids already ascending with the position (rank = position);
//   * a rank table, position of the r-th smallest id at table[r].  Up to
//     COMPARE_MAX ids: by comparisons (the rank of an id is the number of
//     smaller ids in the list); up to RANK_WARP_MAX =
//     32 * RC: a stable LSD radix sort of (id, position) pairs by 8-bit digits
//     of id - (smallest id), by the cell's warp in its shared memory; longer
//     lists: the same sort by a block of k_rank_tables (before k_collide), in
//     shared memory up to RANK_BLOCK_MAX ids and in the scratch buffers above
//     that;
//   * few lookups in a long list: a select per lookup over the list in global
//     memory (select8).
// A block's table of the list at slots [b, b + n) is written to table[b, b + n).

constexpr int RC = 8;                           // rows of 32 ids a warp sorts itself
constexpr uint32_t COMPARE_MAX = 64;            // ids whose ranks come from comparisons
constexpr uint32_t RANK_BLOCK_MAX = 12288;      // longest list the large kernel sorts in shared memory
constexpr int RT_THREADS = 1024;                // threads of a large-kernel block
constexpr uint32_t RT_SEG = 128;                // ids of a warp in a block's sort, at least
constexpr int RT_MID_THREADS = 256;             // threads of a mid-size-kernel block
constexpr int RT_MID_BLOCKS_PER_SM = 5;
constexpr uint32_t SENTINEL = 0xFFFFFFFFu;

struct IdList {
    const uint32_t* table;           // rank -> position, or null
    const uint32_t* base;            // the ids in global memory (select8)
    int top;                         // highest set bit of any id (select8)
    uint32_t n;
    bool sorted;                     // ids ascend with the position: rank = position
};

// lookups up to which a list longer than 32 * RC ids is searched per lookup
// (select8) instead of being sorted into a rank table: a select costs a few
// sweeps of the list by one warp, a table a few sweeps by a whole block
constexpr uint32_t SELECT_LOOKUPS = 4;

// The lanes of the warp whose 8-bit digit d equals this lane's (v: the
// lane holds a digit at all; lanes without one group with none), from nine
// ballots (a warp multisplit).
__device__ __forceinline__ unsigned digit_peers(uint32_t d, bool v) {
    unsigned peers = __ballot_sync(FULL, v);
    peers = v ? peers : ~peers;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool bit = (d >> b) & 1u;
        const unsigned bb = __ballot_sync(FULL, bit);
        peers &= bit ? bb : ~bb;
    }
    return peers;
}

// Position of the rank-th smallest of the n (unique) ids at ids[0, n) by
// one warp: passes over windows of 8 bits from bit `top` (every id is below
// 2^(top + 1)) down, each counting, in the warp's 256 shared counters, the
// ids that share the bits found so far; SENTINEL if rank >= n.  The first
// window is the top 8 bits, so that its digits spread over the counters
// (windows aligned to bit 0 would leave the first pass one or two digits:
// every id's atomic on the same counters); the last window holds the bits
// that remain.  Each lane keeps eight loads in flight.
__device__ __noinline__ uint32_t select8(const uint32_t* __restrict__ ids, uint32_t n, uint32_t rank, int top, uint32_t* cnt,
                            int lane) {
    uint32_t prefix = 0, want = rank;
#pragma unroll 1
    for (int lo = top - 7;; lo -= 8) {
        const int sh = lo > 0 ? lo : 0;
        const int width = lo >= 0 ? 8 : 8 + lo;        // bits of this window
        const uint32_t dm = (1u << width) - 1u;
        const uint32_t hm = sh + width >= 32 ? 0u : (0xFFFFFFFFu << (sh + width));
#pragma unroll
        for (int k = 0; k < 8; ++k) cnt[lane * 8 + k] = 0u;
        __syncwarp();
#pragma unroll 1
        for (uint32_t q0 = 0; q0 < n; q0 += 256) {
            uint32_t x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const uint32_t q = q0 + 32u * u + (uint32_t)lane;
                x[u] = q < n ? ids[q] : 0u;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const uint32_t q = q0 + 32u * u + (uint32_t)lane;
                if (q < n && (x[u] & hm) == prefix) atomicAdd(&cnt[(x[u] >> sh) & dm], 1u);
            }
        }
        __syncwarp();
        uint32_t c[8], sum = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            c[k] = cnt[lane * 8 + k];
            sum += c[k];
        }
        uint32_t xs = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, xs, o);
            if (lane >= o) xs += y;
        }
        const uint32_t before = xs - sum;
        const bool mine = want >= before && want < xs;
        uint32_t d = 0, rest = 0, run = before;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (mine && want >= run && want < run + c[k]) {
                d = (uint32_t)(lane * 8 + k);
                rest = want - run;
            }
            run += c[k];
        }
        const unsigned b = __ballot_sync(FULL, mine);
        __syncwarp();
        if (!b) return SENTINEL;
        const int src = __ffs(b) - 1;
        d = __shfl_sync(FULL, d, src);
        want = __shfl_sync(FULL, rest, src);
        prefix |= d << sh;
        if (sh == 0) break;
    }
    uint32_t pos = SENTINEL;
#pragma unroll 1
    for (uint32_t q0 = 0; q0 < n; q0 += 256) {
        uint32_t x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t q = q0 + 32u * u + (uint32_t)lane;
            x[u] = q < n ? ids[q] : 0u;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t q = q0 + 32u * u + (uint32_t)lane;
            if (q < n && x[u] == prefix && q < pos) pos = q;
        }
    }
    return __reduce_min_sync(FULL, pos);
}

// Scratch of the rank tables, arrays indexed by slot: two (key, value) pair
// buffers and the tables.  They are the sort's other buffer, unused between
// the scatter and the next step's scatter; a list at slots [b, b + n) uses
// [b, b + n) of each.
struct RankScratch {
    uint32_t *xk, *xv, *yk, *yv, *table;
};

// One stable counting pass of an LSD radix sort over the pairs [0, n) by the
// first nw warps of the group (one warp: BLOCK false; the whole block:
// BLOCK true, all threads calling): warp w takes the w-th run of `seg`
// pairs.  Keys come from sk, values from sv (null: the position itself);
// the pairs go to (dk, dv) ordered by the digit (key >> sh) & 255, pairs of
// equal digits keeping their order (dk null: values only).  Per 32 pairs,
// digit_peers groups equal digits; a group's members take consecutive
// places after the digit's running offset in lane order and the group's
// highest lane advances it.  cnt: 256 counters per warp; tot: 256 (BLOCK).
template <bool BLOCK>
__device__ void radix_pass(const uint32_t* sk, const uint32_t* sv, uint32_t* dk, uint32_t* dv, uint32_t n, int sh,
                           int nw, uint32_t* cnt, uint32_t* tot, uint32_t tid, int lane, int w) {
    const uint32_t seg = (n + 32u * nw - 1) / (32u * nw) * 32u;
    const uint32_t q0 = min(n, (uint32_t)w * seg), q1 = min(n, q0 + seg);
    uint32_t* c = cnt + (BLOCK ? w * 256 : 0);
#pragma unroll
    for (int k = 0; k < 8; ++k) c[lane * 8 + k] = 0u;
    __syncwarp();
#pragma unroll 1
    for (uint32_t g = q0; g < q1; g += 32) {
        const uint32_t q = g + lane;
        const uint32_t d = q < q1 ? (sk[q] >> sh) & 255u : 256u;
        const unsigned peers = digit_peers(d, q < q1);
        if (q < q1 && lane == 31 - __clz((int)peers)) c[d] += (uint32_t)__popc(peers);
        __syncwarp();
    }
    // offsets: digit-major over the warps
    if (BLOCK) {
        __syncthreads();
        if (tid < 256) {
            uint32_t run = 0;
            for (int v = 0; v < nw; ++v) {
                const uint32_t x = cnt[v * 256 + tid];
                cnt[v * 256 + tid] = run;
                run += x;
            }
            tot[tid] = run;
        }
        __syncthreads();
    }
    if (!BLOCK || w == 0) {
        uint32_t* t = BLOCK ? tot : c;
        uint32_t cc[8], sum = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            cc[k] = t[lane * 8 + k];
            sum += cc[k];
        }
        uint32_t x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        uint32_t run = x - sum;
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            t[lane * 8 + k] = run;
            run += cc[k];
        }
        __syncwarp();
    }
    if (BLOCK) {
        __syncthreads();
        if (tid < 256)
            for (int v = 0; v < nw; ++v) cnt[v * 256 + tid] += tot[tid];
        __syncthreads();
    }
    unsigned lt;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
#pragma unroll 1
    for (uint32_t g = q0; g < q1; g += 32) {
        const uint32_t q = g + lane;
        const bool in = q < q1;
        const uint32_t key = in ? sk[q] : 0u, val = in ? (sv ? sv[q] : q) : 0u;
        const uint32_t d = in ? (key >> sh) & 255u : 256u;
        const unsigned peers = digit_peers(d, in);
        const uint32_t b = in ? c[d] : 0u;
        __syncwarp();
        if (in) {
            if (lane == 31 - __clz((int)peers)) c[d] = b + (uint32_t)__popc(peers);
            const uint32_t dst = b + (uint32_t)__popc(peers & lt);
            if (dk) dk[dst] = key;
            dv[dst] = val;
        }
        __syncwarp();
    }
    if (BLOCK) __syncthreads();
    else __syncwarp();
}

// Rank table of the n ids staged in xk (unique; highest set bit `top`):
// the digits up to `top`, passes alternating between (yk, yv) and (xk, xv),
// the last one writing the positions to table.
template <bool BLOCK>
__device__ void radix_table(uint32_t n, int top, uint32_t* xk, uint32_t* xv, uint32_t* yk, uint32_t* yv,
                            uint32_t* table, int nw, uint32_t* cnt, uint32_t* tot, uint32_t tid, int lane, int w) {
    const int passes = top / 8 + 1;
    const uint32_t *sk = xk, *sv = nullptr;
#pragma unroll 1
    for (int p = 0; p < passes; ++p) {
        const bool last = p + 1 == passes;
        uint32_t* dk = last ? nullptr : ((p & 1) ? xk : yk);
        uint32_t* dv = last ? table : ((p & 1) ? xv : yv);
        radix_pass<BLOCK>(sk, sv, dk, dv, n, 8 * p, nw, cnt, tot, tid, lane, w);
        sk = dk;
        sv = dv;
    }
}

// Rank tables of the lists that k_collide will use and k_ncand queued for
// this kernel (entries cell << 3 | species bin 0..6; *nq of them, at most
// max_q): one list per block at a time, NT threads, sorted in shared memory
// up to MAXN ids and in the scratch buffers above that.  A list already in
// ascending id order gets the identity.  Passes of the sort bound it: the digits
// are those of id - (smallest id), one or two for most cells where the id itself
// has three, and a warp takes at least RT_SEG ids (64 to 128 alike, 256: 97 us):
// 6200 lists of 257 to 2048 ids 135 -> 90 us, the longer ones 20.6 -> 14.6 us.
template <int NT, uint32_t MAXN>
__global__ void __launch_bounds__(NT) k_rank_tables(const uint32_t* __restrict__ ids, RankScratch S,
                                                    const uint32_t* __restrict__ off, const uint32_t* __restrict__ cnt,
                                                    const uint32_t* __restrict__ q,
                                                    const uint32_t* nq, uint32_t max_q, uint32_t C,
                                                    const DevState* st) {
    if (block_faulted(st)) return;                   // a fault was flagged: the state is not stepped further
    constexpr int NWARPS = NT / 32;
    extern __shared__ uint32_t s_buf[];                 // four arrays of MAXN
    __shared__ uint32_t s_cnt[NWARPS * 256];
    __shared__ uint32_t s_tot[256];
    __shared__ uint32_t s_lo[NWARPS], s_hi[NWARPS];
    const uint32_t nb = min(*nq, max_q);             // an overflow is flagged by k_ncand
    const uint32_t tid = threadIdx.x;
    const int lane = (int)(tid & 31u), w = (int)(tid >> 5);
    for (uint32_t b = blockIdx.x; b < nb; b += gridDim.x) {
        const uint32_t e = q[b];
        const uint32_t bin = (e & 7u) * C + (e >> 3);
        const uint32_t slot0 = off[bin], n = cnt[bin];
        const uint32_t* base = ids + slot0;
        const bool in_smem = n <= MAXN;
        uint32_t* xk = in_smem ? s_buf : S.xk + slot0;
        uint32_t* xv = in_smem ? s_buf + MAXN : S.xv + slot0;
        uint32_t* yk = in_smem ? s_buf + 2 * MAXN : S.yk + slot0;
        uint32_t* yv = in_smem ? s_buf + 3 * MAXN : S.yv + slot0;
        uint32_t* table = S.table + slot0;
        uint32_t lo = 0xFFFFFFFFu, hi = 0u;
        for (uint32_t k = tid; k < n; k += NT) {
            const uint32_t x = base[k];
            xk[k] = x;
            lo = min(lo, x);
            hi = max(hi, x);
        }
        lo = __reduce_min_sync(FULL, lo);
        hi = __reduce_max_sync(FULL, hi);
        if (lane == 0) {
            s_lo[w] = lo;
            s_hi[w] = hi;
        }
        __syncthreads();
        bool asc = true;
        for (uint32_t k = tid; k + 1 < n; k += NT)
            if (!(xk[k] < xk[k + 1])) asc = false;
        if (__syncthreads_and(asc)) {
            for (uint32_t r = tid; r < n; r += NT) table[r] = r;
        } else {
#pragma unroll
            for (int v = 0; v < NWARPS; ++v) {
                lo = min(lo, s_lo[v]);
                hi = max(hi, s_hi[v]);
            }
            for (uint32_t k = tid; k < n; k += NT) xk[k] -= lo;
            __syncthreads();
            const int top = hi > lo ? 31 - __clz((int)(hi - lo)) : 0;
            const int nw = (int)min((uint32_t)NWARPS, (n + RT_SEG - 1u) / RT_SEG);
            radix_table<true>(n, top, xk, xv, yk, yv, table, nw, s_cnt, s_tot, tid, lane, w);
        }
        __syncthreads();
    }
}

// Ranks of the n <= RANK_WARP_MAX ids at base, `lookups` of which follow, by
// one warp.  Returns 0 when the ids ascend, 1 when table[0, n) was written, 2 when
// select8 costs less (never with want_table).  sbuf: four arrays of
// RANK_WARP_MAX, then 256 counters.  Out of line: one copy serves every list.
//
// Costs in instructions: comparing n ids 13 n / 4 per 32 of them, a radix pass 96 +
// 64 per 32 ids, a select8 pass 130; but the comparisons are one short loop where
// the sort's code is fetched anew for nearly every list (stress case, 685 -> 520
// us with 64 ids by comparison; 128 the same, 256 slower).  A cell's own heavies
// have neighbouring ids, so that the digits of id - (smallest id), not of the id,
// decide the passes: a cell of 80 atoms takes one or two instead of four.
__device__ __noinline__ int rank_list(const uint32_t* __restrict__ base, uint32_t n, uint32_t lookups, uint32_t* table,
                                      uint32_t* sbuf, int id_top, bool want_table) {
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t* xk = sbuf;
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
    const uint32_t n4 = (n + 127u) & ~127u;
    __syncwarp();                                // the buffer's last readers are done
#pragma unroll 1
    for (uint32_t q0 = 0; q0 < n4; q0 += 128) {
        uint32_t x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t q = q0 + 32u * k + lane;
            x[k] = q < n ? base[q] : 0xFFFFFFFFu;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t q = q0 + 32u * k + lane;
            xk[q] = x[k];                        // (ids are below 2^32 - 1: the rest sorts last)
            if (q < n) {
                lo = min(lo, x[k]);
                hi = max(hi, x[k]);
            }
        }
    }
    __syncwarp();
    bool asc = true;
#pragma unroll 1
    for (uint32_t q = lane; q + 1 < n; q += 32)
        if (!(xk[q] < xk[q + 1])) asc = false;
    if (__all_sync(FULL, asc)) return 0;
    lo = __reduce_min_sync(FULL, lo);
    hi = __reduce_max_sync(FULL, hi);
    const int top = hi > lo ? 31 - __clz((int)(hi - lo)) : 0;
    const uint32_t passes = (uint32_t)(top / 8 + 1);
    if (n <= COMPARE_MAX) {
        const uint4* x4 = reinterpret_cast<const uint4*>(xk);
#pragma unroll 1
        for (uint32_t q = lane; q < ((n + 31u) & ~31u); q += 32) {
            const uint32_t a = xk[q];
            uint32_t r = 0;
#pragma unroll 1
            for (uint32_t j = 0; 4u * j < n; ++j) {
                const uint4 v = x4[j];
                r += (v.x < a ? 1u : 0u) + (v.y < a ? 1u : 0u) + (v.z < a ? 1u : 0u) + (v.w < a ? 1u : 0u);
            }
            if (q < n) table[r] = q;
        }
        __syncwarp();
        return 1;
    }
    const uint32_t tab_cost = passes * (96u + ((n + 31u) / 32u) * 64u);
    if (!want_table && lookups * (uint32_t)(id_top / 8 + 2) * 130u < tab_cost) return 2;
#pragma unroll 1
    for (uint32_t q = lane; q < n; q += 32) xk[q] -= lo;
    __syncwarp();
    radix_table<false>(n, top, xk, sbuf + RANK_WARP_MAX, sbuf + 2 * RANK_WARP_MAX, sbuf + 3 * RANK_WARP_MAX, table, 1,
                       sbuf + 4 * RANK_WARP_MAX, nullptr, lane, (int)lane, 0);
    return 1;                                    // ordered for the warp by radix_pass's final __syncwarp
}

// ids of one cell and species at slots [slot0, slot0 + n), `lookups` rank
// selections to follow; stab: where a table of the warp's own goes
__device__ __forceinline__ void load_ids(IdList& L, const uint32_t* __restrict__ ids, uint32_t slot0, uint32_t n,
                                         uint32_t lookups, const RankScratch& S, uint32_t* sbuf, uint32_t* stab,
                                         int id_top, bool want_table = false) {
    L.n = n;
    L.base = ids + slot0;
    L.top = id_top;
    L.table = nullptr;
    L.sorted = false;
    if (n > 32u * RC) {
        // a table built by k_rank_tables, or few lookups
        if (want_table || lookups > SELECT_LOOKUPS) L.table = S.table + slot0;
        return;
    }
    const int how = rank_list(L.base, n, lookups, stab, sbuf, id_top, want_table);
    L.sorted = how == 0;
    if (how == 1) L.table = stab;
}

// A cell of this many candidates is taken by a block of k_collide: one warp would
// still be at it when all others are done (candidates go with the square of the
// density: 1300 in one cell where the average has three; 920 us with a warp, 541
// with a block; lines at 64, 128 and 256 within 3 % of each other).
constexpr uint32_t BIG_CELL = 256;
constexpr uint32_t BIG_FLAG = 0x80000000u;      // (cells are below 2^24)

// Heavy cells (a list the warp must sort or many candidates) go to the
// front of `active`, the others to its back, so that k_collide starts them
// first.
// EXT: any of the step-wise, heavy-pair or Coulomb extensions is on (the
// plain variant counts the classes (e, Cu) and (e, Cu+) only)
template <bool EXT>
__global__ void __launch_bounds__(256) k_ncand(const uint32_t* __restrict__ cnt, const float* __restrict__ ck,
                                               uint4* nc, uint4* nc2, uint32_t* cand, uint32_t* active, uint32_t* mid,
                                               uint32_t* big, DevState* st, KParams P) {
    if (st->error) return;                           // a fault was flagged: the state is not stepped further
    const uint32_t C = P.ncell;
    const int lane = threadIdx.x & 31;
    const uint32_t stride = gridDim.x * blockDim.x;
    const bool heavy_pairs = EXT && P.heavy_coll && P.heavy_step;
    const bool q3 = EXT && P.charge_max >= 3, q4 = EXT && P.charge_max >= 4;
    for (uint32_t c0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); c0 < C; c0 += stride) {
        const uint32_t c = c0 + lane;
        // n[k]: candidates of class k (electron classes 0-4, heavy pairs 5, 6)
        uint32_t n[NCLS] = {0, 0, 0, 0, 0, 0, 0};
        uint32_t N[NSP] = {0, 0, 0, 0, 0, 0, 0};
        int r = -1;
        if (c < C) {
            // list lengths (Cu3+ and Cu4+ have bins with charge_max >= 3; Cu4+ is
            // drawn only by the Coulomb pairs)
#pragma unroll
            for (int sp = 0; sp < NSP; ++sp)
                if ((sp < 5 || q3) && (sp < 6 || P.coulomb)) N[sp] = cnt[sp * C + c];
            const uint32_t Nt[NECLS] = {N[SP_CU], N[SP_CUP], N[SP_CU2_SW], N[SP_CU2_DI], N[SP_CU3]};
            bool ecls = false;
            for (int k = 0; k < NECLS; ++k) ecls |= Nt[k] > 0;
            ecls = ecls && N[SP_E] > 0;
            const bool hcls = heavy_pairs && N[SP_CU] > 0;
            if (ecls || hcls) {
                r = run_of(P, c);
                const RunInfo& RI = P.runs[r];
                const uint32_t lc = c - RI.cell_base;
                const uint32_t j = lc % (uint32_t)RI.nr;
                // the cell's stream gives R_k to class k whether the class is on or not
                Stream s(lc, st->step, SID_NCAND, RI.seed, RI.run);
                float R[NCLS];
#pragma unroll
                for (int k = 0; k < NCLS; ++k) R[k] = s.u01();
                if (ecls) {
#pragma unroll
                    for (int k = 0; k < NECLS; ++k) {
                        if (k >= 2 && !q3) break;
                        if (k == 4 && !q4) break;
                        const float x = ((float)N[SP_E] * (float)Nt[k]) * ck[RI.ck_base + k * RI.nr + j] + R[k];
                        n[k] = (uint32_t)floorf(x);
                    }
                }
                if (hcls) {
                    // N_cu N_cu+ charge-exchange pairs, N_cu (N_cu - 1) / 2 Cu-Cu
                    // pairs (the 1/2 is in the row factor)
                    const uint32_t Ncu = N[SP_CU], Ni = N[SP_CUP];
                    const float x5 = ((float)Ncu * (float)Ni) * ck[RI.ck_base + 5 * RI.nr + j] + R[5];
                    const float x6 = ((float)Ncu * (float)(Ncu - 1u)) * ck[RI.ck_base + 6 * RI.nr + j] + R[6];
                    n[5] = (uint32_t)floorf(x5);
                    n[6] = Ncu >= 2 ? (uint32_t)floorf(x6) : 0u;
                }
            }
            nc[c] = make_uint4(n[0], n[1], n[5], n[6]);
            if (q3) nc2[c] = make_uint4(n[2], n[3], n[4], 0u);
            cand[c] = n[0] + n[1] + n[2] + n[3] + n[4];    // the electron classes reserve spawn slots
        }
        // heavy candidates join the run's candidate count here (the electron
        // classes' are summed from the spawn-slot scan)
        const uint32_t nh = n[5] + n[6];
        if (__any_sync(FULL, nh > 0)) {
            const int r0 = __shfl_sync(FULL, r, 0);
            if (__all_sync(FULL, nh == 0 || r == r0)) {
                const uint32_t t = __reduce_add_sync(FULL, nh);
                if (lane == 0) atomicAdd(&P.rs[r0].ctr[C_CAND], (unsigned long long)t);
            } else if (nh > 0) {
                atomicAdd(&P.rs[r].ctr[C_CAND], (unsigned long long)nh);
            }
        }
        // lookups of each species' list over the classes that draw from it;
        // the Coulomb pairs look up every electron and every ion of a cell
        // with electrons (k_collide counts the same)
        uint32_t look[NSP];
        look[SP_E] = n[0] + n[1] + n[2] + n[3] + n[4];
        look[SP_CU] = n[0] + n[5] + 2u * n[6];
        look[SP_CUP] = n[1] + n[5];
        look[SP_CU2_SW] = n[2];
        look[SP_CU2_DI] = n[3];
        look[SP_CU3] = n[4];
        look[SP_CU4] = 0;
        uint32_t ncoul = 0;          // Coulomb pairs of the cell (about)
        if (EXT && P.coulomb && N[SP_E] > 0) {
            look[SP_E] += N[SP_E];
            ncoul = N[SP_E] / 2u;
#pragma unroll
            for (int sp = SP_CUP; sp < NSP; ++sp) ncoul += N[sp] > 0 ? max(N[SP_E], N[sp]) : 0u;
        }
        // the ion lists: with electrons, or on heavy steps (ion pairs)
        if (EXT && P.coulomb && (N[SP_E] > 0 || P.heavy_step)) {
#pragma unroll
            for (int sp = SP_CUP; sp < NSP; ++sp) {
                look[sp] += N[sp];
                ncoul += P.heavy_step ? N[sp] : 0u;
            }
        }
        // k_collide takes the cells with DSMC candidates; k_coulomb visits the
        // others itself, but the rank tables it needs are queued here too
        const uint32_t ntot = n[0] + n[1] + n[2] + n[3] + n[4] + nh;
        const bool act = c < C && ntot > 0;
        const uint32_t RL = 32u * RC;
        bool long_list = false;
#pragma unroll
        for (int sp = 0; sp < NSP; ++sp) long_list |= look[sp] > 0 && N[sp] > RL;
        const bool heavy = act && (ntot > 32u || long_list);
        unsigned lt;
        asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
        const unsigned mh = __ballot_sync(FULL, heavy), ml = __ballot_sync(FULL, act && !heavy);
        uint32_t bh = 0, bl = 0;
        if (mh && lane == __ffs(mh) - 1) bh = atomicAdd(&st->n_heavy, (uint32_t)__popc(mh));
        if (ml && lane == __ffs(ml) - 1) bl = atomicAdd(&st->n_light, (uint32_t)__popc(ml));
        if (mh) bh = __shfl_sync(FULL, bh, __ffs(mh) - 1);
        if (ml) bl = __shfl_sync(FULL, bl, __ffs(ml) - 1);
        if (heavy) active[bh + __popc(mh & lt)] = ntot >= BIG_CELL ? c | BIG_FLAG : c;
        else if (act) active[C - 1u - (bl + __popc(ml & lt))] = c;
        if (act || (c < C && ncoul > 0)) {
            // the lists k_collide or k_coulomb will rank that need a block's
            // sort (long, with more lookups than select8 serves)
            for (uint32_t sp = 0; sp < (uint32_t)NSP; ++sp) {
                if (look[sp] == 0 || N[sp] <= RANK_WARP_MAX || look[sp] <= SELECT_LOOKUPS) continue;
                const bool large = N[sp] > RANK_MID_MAX;
                const uint32_t x = atomicAdd(large ? &st->n_big : &st->n_mid, 1u);
                if (x < rank_queue_max(P.capacity, large ? RANK_MID_MAX : RANK_WARP_MAX))
                    (large ? big : mid)[x] = (c << 3) | sp;
                else set_error(st, ERR_BOUNDS);
            }
        }
    }
}

// cross sections of a pair: running sums cum[] of the class's channels at
// the pair's relative energy, and sigma_T g
struct PairEval {
    float cum[4];
    float sg;
};

// pair classes: first channel and target species of class k (the electron
// classes draw an electron as the first particle, the heavy pairs a Cu)
__device__ __forceinline__ int class_ch0(int k) {
    return k == 0 ? CH_EL : k == 1 ? CH_SW : k <= 3 ? CH_S3 : k == 4 ? CH_S4 : k == 5 ? CH_CX : CH_NN;
}
__device__ __forceinline__ int class_target(int k) {
    return k == 0 ? SP_CU : k == 1 ? SP_CUP : k == 2 ? SP_CU2_SW : k == 3 ? SP_CU2_DI : k == 4 ? SP_CU3
         : k == 5 ? SP_CUP : SP_CU;
}

__device__ __forceinline__ PairEval evaluate_pair(int k, const V3& ve, const V3& vt, const float* __restrict__ xsE,
                                                  const float* __restrict__ xs, const CollConsts& cc) {
    PairEval e;
    const float ux = ve.x - vt.x, uy = ve.y - vt.y, uz = ve.z - vt.z;
    const float g2 = (ux * ux + uy * uy) + uz * uz;
    const float g = sqrtf(g2);
    const float eps = g2 * (k < NECLS ? cc.kmr : cc.kmr_h);
    const int ch0 = class_ch0(k);
    const int nch = k == 0 ? 4 : 1;
    float sT = 0.0f;
    for (int q = 0; q < 4; ++q) {
        if (q < nch) sT = sT + xs_lookup(xsE, xs + (ch0 + q) * XS_N, eps);
        e.cum[q] = sT;
    }
    e.sg = sT * g;
    return e;
}

// a pair whose particles are no longer what its class draws: a target
// ionized earlier this step or, for the heavy classes, a Cu that was
__device__ __forceinline__ bool consumed_pair(int k, uint32_t akey, uint32_t tkey) {
    const int ts = class_target(k);
    const bool t_gone = (tkey & KEY_FLAG) || (int)key_species(tkey) != ts;
    if (k < NECLS) return t_gone;
    return t_gone || (akey & KEY_FLAG) || (int)key_species(akey) != SP_CU;
}

// What became of a candidate: a channel's event (its channel), or one of these
// (indices of a warp's counters).
enum { OUT_NULL = NCH, OUT_CONSUMED, OUT_THR, OUT_VIOL, OUT_FB, OUT_N };
constexpr int COLL_WARPS = 4;                   // warps of a k_collide block
constexpr int COLL_SORT_WORDS = 4 * RANK_WARP_MAX + 256;
constexpr uint32_t CLAIMS = 4 * RANK_WARP_MAX;  // places of a block's claim tables (in the rank buffers of its warps 1 and 2)
// a spawned electron (its position is a particle's of the pair)
struct Spawn {
    uint32_t cell;
    float pz, pr;
    V3 v;
};

// One candidate of class k on particles ie (electron, or Cu of a heavy pair) and
// it, by its lane: target and acceptance tests, channel, kinematics, the
// particles' new state and the target's charge.  Returns the outcome; `viol`: the
// pair broke the majorant; the electrons it makes (nsp of them, in order) go to
// sp[], to be placed by the caller in candidate order.
template <bool EXT>
__device__ __forceinline__ int collide_pair(Particles& A, int k, uint32_t ie, uint32_t it, uint32_t lc, uint32_t m,
                                            float Racc, float Rch, const RunInfo* RI, int geom,
                                            const float* __restrict__ xsE, const float* __restrict__ xs,
                                            const CollConsts& cc, const DevState* st, long long* rho_h, bool& viol,
                                            uint32_t& fb, int& nsp, Spawn (&sp)[2]) {
    const uint32_t tkey = A.key[it];
    const uint32_t akey = EXT && k >= NECLS ? A.key[ie] : 0u;
    V3 ve{A.vz[ie], A.vr[ie], A.vt[ie]}, vt{A.vz[it], A.vr[it], A.vt[it]};
    const PairEval ev = evaluate_pair(k, ve, vt, xsE, xs, cc);
    if (consumed_pair(k, akey, tkey)) return OUT_CONSUMED;       // ionized (or charged) earlier this step
    viol = ev.sg > cc.sgmax[k];
    if (!(Racc * cc.sgmax[k] < ev.sg)) return OUT_NULL;
    if (EXT && k == 5) {
        // charge exchange Cu + Cu+ -> Cu+ + Cu moves the electron, not the
        // atoms: each slot keeps its species and takes the other's velocity
        A.vz[ie] = vt.x; A.vr[ie] = vt.y; A.vt[ie] = vt.z;
        A.vz[it] = ve.x; A.vr[it] = ve.y; A.vt[it] = ve.z;
        return CH_CX;
    }
    // channel: the first whose running sum exceeds Rch sigma_T (else the last
    // with a cross section)
    const int nch = k == 0 ? 4 : 1;
    const float r = Rch * ev.cum[3];
    int q = -1, last = nch - 1;
#pragma unroll
    for (int a = 3; a >= 0; --a)
        if (a < nch && r < ev.cum[a]) q = a;
    if (q < 0) {
        bool found = false;
#pragma unroll
        for (int a = 3; a >= 0; --a)
            if (!found && a < nch && ev.cum[a] > (a ? ev.cum[a > 0 ? a - 1 : 0] : 0.0f)) {
                last = a;
                found = true;
            }
        q = last;
    }
    const int ch = class_ch0(k) + q;
    const bool ionizes = ch != CH_EL && ch != CH_EXC && ch != CH_NN;
    // the candidate's stream after its four pair-choice draws
    StreamOf<true> rs(lc, st->step, sid_cand(k, m), RI->seed, RI->run);
    rs.ctr.w = 1u;
    // Stage 1, Eq. (12): the pair scatters and loses the channel's energy (a Cu
    // pair elastically, equal masses); stage 3, Eq. (14), of an ionization: e1 + e2
    // elastic, e2 born with the velocity of A* (stage 2, Eq. (13))
    V3 a = ve, b = vt;
    float kth = ch == CH_EL || ch == CH_NN ? 0.0f : cc.kth[ch];
    float a1 = ch == CH_NN ? 0.5f : cc.a_e, a2 = ch == CH_NN ? 0.5f : cc.a_t;
#pragma unroll 1
    for (int stage = 0;; ++stage) {
        if (!binary_scatter(rs, a, b, kth, a1, a2, fb)) return OUT_THR;
        if (stage == 0) vt = b;
        if (stage == 1 || !ionizes) break;
        kth = 0.0f;
        a1 = a2 = 0.5f;
    }
    ve = a;
    if (ionizes) {
        const uint32_t tcell = key_cell(tkey);
        const int ts = class_target(k);
        const int new_sp = ch == CH_SI ? SP_CUP : ch == CH_SW ? SP_CU2_SW : ch == CH_DI ? SP_CU2_DI
                         : ch == CH_S3 ? SP_CU3 : SP_CU4;
        const float tpz = A.pz[it], tpr = A.pr[it];
        sp[0] = Spawn{tcell, tpz, tpr, b};
        nsp = 1;
        if (ch == CH_DI) {
            // Stage 4, Eq. (15): e3 -> e5 + e6 (velocity rectangle)
            V3 e5, e6;
            rectangle_split(rs, ve, e5, e6, cc.di_split_mode, fb);
            sp[1] = Spawn{key_cell(A.key[ie]), A.pz[ie], A.pr[ie], e6};
            nsp = 2;
            ve = e5;
        }
        A.key[it] = converted_key((uint32_t)new_sp, (uint32_t)ts, tcell);
        deposit1(rho_h, *RI, geom, tcell - RI->cell_base, tpz, tpr, charge_of(new_sp) - charge_of(ts));
    }
    A.vz[ie] = ve.x; A.vr[ie] = ve.y; A.vt[ie] = ve.z;
    A.vz[it] = vt.x; A.vr[it] = vt.y; A.vt[it] = vt.z;
    return ch;
}

// ---------------------------------------------------------------------
// Coulomb collisions (listed by Sec. 2.3 without a method): the binary
// collision model of Takizuka and Abe (1977).  A pair with relative velocity
// u turns by theta, tan(theta / 2) = delta, delta = sqrt(Kn / u^3) Z with Z
// normal (here the Irwin-Hall sum of twelve uniforms), about a uniform
// azimuth; |u| is kept and the change is shared by the reduced mass.  Kn =
// (q_a q_b)^2 n_L lnL dt / (8 pi eps0^2 m_ab^2).  The float operations are
// those of the oracle's float build, in the same order.
//
// A pair's particles and random numbers do not depend on any velocity: the
// particles come from keyed permutations of the id ranks, and each pair
// draws from a stream of its own (twelve uniforms for Z, then the azimuth).
// So a warp first derives them for 32 pairs at a time, flattened over all the
// classes of a batch of cells, and then applies the pairs in rounds: in each, the
// pairs whose earlier sharers of a particle are through (by the sequential
// definition the regular pairs of a species with itself share none, the three of
// an odd count's closing triple do, and each pair of two species does with the
// one N_fewer pairs before it).
// ---------------------------------------------------------------------

// Pseudo-random permutation of [0, n): four Feistel rounds (Luby and Rackoff)
// on 2h bits, 4^h >= n, with an integer mixing round function, walked back
// into [0, n) by cycle walking (Black and Rogaway, 2002).  The walk ends
// within 4^h steps because x itself lies in [0, n).
__device__ __forceinline__ uint32_t fe_round(uint32_t x, uint32_t k) {
    uint32_t t = (x ^ k) * 0x9E3779B1u;
    t ^= t >> 15;
    t *= 0x85EBCA77u;
    t ^= t >> 13;
    return t;
}
// h of the permutation of [0, n): the least h >= 1 with 4^h >= n
__device__ __forceinline__ int perm_bits(uint32_t n) {
    return n > 4u ? (33 - __clz((int)(n - 1u))) / 2 : 1;
}
// one pass of the four Feistel rounds on 2h bits
__device__ __forceinline__ uint32_t feistel4(uint32_t y, const uint4& key, int h) {
    const uint32_t mask = (1u << h) - 1u;
    uint32_t L = y >> h, R = y & mask;
    const uint32_t k4[4] = {key.x, key.y, key.z, key.w};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const uint32_t F = fe_round(R, k4[r]) & mask;
        const uint32_t t = L ^ F;
        L = R;
        R = t;
    }
    return (L << h) | R;
}
// Indices x0 and x1 under two permutations (or the same one twice), each
// walked back into its range [0, n) by repeating the rounds until the value
// falls in it, one walk after the other in one loop: a warp then takes as many
// rounds as its longest pair of walks has (side by side it took twice the longest
// walk's: k_coulomb 475 -> 417 us with that and 32-bit counts).
// A walk ends within 4^h steps, x lying in [0, n) itself (x is returned after
// 4^h, which it never reaches).
__device__ void perm_index2(uint32_t x0, uint32_t n0, const uint4& key0, int h0, uint32_t x1, uint32_t n1,
                            const uint4& key1, int h1, uint32_t& out0, uint32_t& out1) {
    out0 = x0;
    out1 = x1;
    uint4 key = key0;
    uint32_t y = x0, n = n0;
    int h = h0;
    bool second = false;
    uint32_t left = h0 < 16 ? 1u << (2 * h0) : 0xFFFFFFFFu;
#pragma unroll 1
    for (;;) {
        y = feistel4(y, key, h);
        const bool in = y < n;
        if (in || --left == 0u) {
            if (second) {
                if (in) out1 = y;
                return;
            }
            if (in) out0 = y;
            second = true;
            key = key1;
            y = x1;
            n = n1;
            h = h1;
            left = h1 < 16 ? 1u << (2 * h1) : 0xFFFFFFFFu;
        }
    }
}

// uniform on [0, 1) from the top 24 bits of a draw (as Stream::u01)
__device__ __forceinline__ float u01_of(uint32_t x) { return __fmul_rn((float)(x >> 8), 5.9604644775390625e-08f); }

// The draws of one Coulomb pair from its stream: Z (the Irwin-Hall sum of
// the first twelve uniforms, three Philox blocks) and the azimuth (points of
// the square from the following blocks, two per block, until one falls in
// the unit disc; fail after 64 tries, as azimuth()).  The three blocks of Z
// and the first block of the azimuth (which serves all but about one pair in
// twenty) are independent chains of rounds, computed side by side.
__device__ void coul_draws(uint32_t subject, uint32_t step, uint32_t sid, uint32_t seed, uint32_t run, float& z,
                           float& c, float& s, bool& fail) {
    const uint2 key = make_uint2(seed, run);
    const uint4 r0 = philox4x32_10(make_uint4(subject, step, sid, 0u), key);
    const uint4 r1 = philox4x32_10(make_uint4(subject, step, sid, 1u), key);
    const uint4 r2 = philox4x32_10(make_uint4(subject, step, sid, 2u), key);
    uint4 r = philox4x32_10(make_uint4(subject, step, sid, 3u), key);
    float zz = 0.0f;
    zz = zz + u01_of(r0.x);
    zz = zz + u01_of(r0.y);
    zz = zz + u01_of(r0.z);
    zz = zz + u01_of(r0.w);
    zz = zz + u01_of(r1.x);
    zz = zz + u01_of(r1.y);
    zz = zz + u01_of(r1.z);
    zz = zz + u01_of(r1.w);
    zz = zz + u01_of(r2.x);
    zz = zz + u01_of(r2.y);
    zz = zz + u01_of(r2.z);
    zz = zz + u01_of(r2.w);
    z = zz - 6.0f;
    fail = false;
#pragma unroll 1
    for (uint32_t b = 0; b < 32u; ++b) {
        if (b > 0u) r = philox4x32_10(make_uint4(subject, step, sid, 3u + b), key);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float u1 = 2.0f * u01_of(h ? r.z : r.x) - 1.0f;
            const float u2 = 2.0f * u01_of(h ? r.w : r.y) - 1.0f;
            const float q = u1 * u1 + u2 * u2;
            if (q < 1.0f && q > 0.0f) {
                const float rq = sqrtf(q);
                c = u1 / rq;
                s = u2 / rq;
                return;
            }
        }
    }
    fail = true;
    c = 1.0f;
    s = 0.0f;
}

// One pair's turn (after its draws): false when u = 0 (nothing to turn).
__device__ __forceinline__ bool coulomb_turn(V3& va, V3& vb, float Kn, float fa, float fb_, float z, float cph,
                                             float sph) {
    const float ux = va.x - vb.x, uy = va.y - vb.y, uz = va.z - vb.z;
    const float u2 = (ux * ux + uy * uy) + uz * uz;
    if (!(u2 > 0.0f)) return false;
    const float u = sqrtf(u2);
    float var = Kn / (u2 * u);
    var = var < 1e30f ? var : 1e30f;                // u -> 0: keep delta finite
    const float d = sqrtf(var) * z;
    // sin(theta) = 2 delta / (1 + delta^2), 1 - cos(theta) = 2 delta^2 / (1 + delta^2)
    float sth, omc;
    const float ad = d < 0.0f ? -d : d;
    if (ad <= 1.0f) {
        const float d2 = d * d, den = 1.0f + d2;
        sth = (2.0f * d) / den;
        omc = (2.0f * d2) / den;
    } else {
        const float rr = 1.0f / d, r2 = rr * rr, den = 1.0f + r2;
        sth = (2.0f * rr) / den;
        omc = 2.0f / den;
    }
    const float sc = sth * cph, ss = sth * sph;
    const float up = sqrtf(ux * ux + uy * uy);
    float dx, dy, dz;
    if (up > 0.0f) {
        const float a1 = ux / up, a2 = uy / up;
        dx = ((a1 * uz) * sc - (a2 * u) * ss) - ux * omc;
        dy = ((a2 * uz) * sc + (a1 * u) * ss) - uy * omc;
        dz = -(up * sc) - uz * omc;
    } else {                                         // u along the third axis
        dx = uz * sc;
        dy = uz * ss;
        dz = -(uz * omc);
    }
    va.x = va.x + fa * dx; va.y = va.y + fa * dy; va.z = va.z + fa * dz;
    vb.x = vb.x - fb_ * dx; vb.y = vb.y - fb_ * dy; vb.z = vb.z - fb_ * dz;
    return true;
}

// Classes of a cell: 0 the electrons with themselves, 1 + i the electrons
// with ion species i (Cu+, Cu2+ SW, Cu2+ DI, Cu3+, Cu4+), on heavy steps
// 6.. the ion species a <= b (in order).  Lists: 0 the electrons, 1 + i ion
// species i.
constexpr int COUL_NCLS = 21;
constexpr int COUL_NLIST = 6;
// A warp's batch of cells: at most 32 classes and 32 lists, and, unless it is one
// cell, COUL_CACHE charged particles, whose velocities the warp holds in shared
// memory (in the words of its rank-table sort buffer, free once the tables are
// built; then COUL_MASKS words of the conflict table)
constexpr int COUL_CACHE = 336, COUL_MASKS = 256;
constexpr int COUL_CELLS = 10;          // most cells of a warp: with electrons and Cu+ their 30 classes fill a batch
constexpr int COUL_BLOCKS = 22;         // blocks (of a warp) an SM
constexpr int COUL_SORT_WORDS = 4 * RANK_WARP_MAX + 256, COUL_CACHE_WORDS = 3 * COUL_CACHE + COUL_MASKS;
constexpr int COUL_SBUF = COUL_SORT_WORDS > COUL_CACHE_WORDS ? COUL_SORT_WORDS : COUL_CACHE_WORDS;

struct CoulClass {
    uint4 k1, k2;          // permutation keys: of the one species; or of the more and the fewer
    float Kn, fa, fb;
    uint32_t P;            // one species: regular pairs; two: the fewer's count (a round)
    uint32_t N;            // one species: its count; two: the more numerous's
    uint32_t lc;           // the cell's index in its run
    uint32_t ba, na, ca;   // the list of a pair's first particle: first slot, count, place in the velocity cache
    uint32_t bb, nb, cb;   // of its second
    uint8_t cls, spa, spb;
    uint8_t flags;         // 1: list a is the more numerous (a on a tie); 2, 4: the ids of list a, b ascend
};
struct CoulWarp {
    CoulClass cl[32];
    uint32_t start[32];                 // a class's first pair in the batch's order
    uint32_t lbase[32], lcoff[32];      // the lists: first slot, place in the cache
};

__device__ __forceinline__ void class_lists(int t, int& la, int& lb) {
    if (t == 0) {
        la = lb = 0;
    } else if (t < 6) {
        la = 0;
        lb = t;
    } else {
        int idx = t - 6, a = 0;
        while (idx >= 5 - a) {
            idx -= 5 - a;
            ++a;
        }
        la = 1 + a;
        lb = 1 + a + idx;
    }
}
__device__ __forceinline__ int list_species(int l) { return l == 0 ? SP_E : SP_CUP + l - 1; }

// The Coulomb pairs (after all cells' DSMC classes: cells are independent,
// so this is the order of cell-by-cell processing), on the lists of the step's
// start; a particle whose species changed this step is left out.
//
// Instructions bound it, and a cell has few pairs (ten to twenty with five
// electrons and five ions).  A warp therefore collects cells (grid-stride) until
// their classes or particles fill its tables and takes all their pairs together, a
// lane a pair: their permutations, draws and lookups side by side, then their turns
// in rounds.  A pair's turn waits for the earlier pairs of the chunk that share a
// particle with it, no others: a pair of lane q sets bit q in the word of each of
// its particles, and the lower bits in its two words are those it waits for (in a
// cell beyond the cache particles share words, and the pairs named are compared).
// Blocks of one warp and up to ten cells keep the SMs evenly loaded (cells differ).
//
// 256 x 512 cells of about eight electrons and eight Cu+ (lognormal), all pairs:
// 826 us and 4060 instructions a cell with a warp a cell, its pairs in the
// classes' waves of disjoint pairs (12.5 threads an instruction); 500 us and 2290
// with batches and rounds; 450-475 us with blocks of one warp, at 22 an SM (20:
// 490 us, 16: 530), 417 us with shorter permutation walks.  Of it the turns take 120
// us, the rank tables 80, the permutations about 120 (their walks differ in length;
// tables of the permutations of up to 16 places took as long to make).
__global__ void __launch_bounds__(32, COUL_BLOCKS) k_coulomb(Particles A, RankScratch S, const uint32_t* __restrict__ off,
                                                   const uint32_t* __restrict__ cnt, DevState* st, KParams P,
                                                   CollConsts cc, const double* __restrict__ cw, uint32_t cells) {
    if (st->error) return;                           // a fault was flagged: the state is not stepped further
    __shared__ __align__(16) uint32_t sbuf[COUL_SBUF];      // rank-table sort, then velocity cache and conflict table
    __shared__ __align__(16) CoulWarp W;
    const int lane = (int)threadIdx.x;
    float* const cvz = reinterpret_cast<float*>(sbuf);
    float* const cvr = cvz + COUL_CACHE;
    float* const cvt = cvr + COUL_CACHE;
    uint32_t* const mask = sbuf + 3 * COUL_CACHE;
    const uint32_t C = P.ncell, step = st->step;
    const uint32_t cell0 = blockIdx.x * cells, cell1 = min(cell0 + cells, C);
    unsigned lt;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
    int la = 0, lb = 0;                               // lane t < COUL_NCLS: the lists of class t
    if (lane < COUL_NCLS) class_lists(lane, la, lb);
    const int lsp = lane < COUL_NLIST ? list_species(lane) : NSP;
    // the batch: run, classes, lists, particles, pairs
    int run = 0, ncl = 0, nlist = 0;
    uint32_t tot = 0, T = 0;
    uint32_t n_ee = 0, n_ei = 0, n_ii = 0, n_fb = 0;
    for (uint32_t c = cell0;; ++c) {
        const bool end = c >= cell1;
        // the cell's charged lists (lane l reads list l)
        uint32_t nl = 0, bl = 0;
        if (!end && lsp < P.nsp) {
            const uint32_t b = (uint32_t)lsp * C + c;
            nl = cnt[b];
            bl = off[b];
        }
        // lane t: class t's pairs
        const uint32_t Na = __shfl_sync(FULL, nl, la), Nb = __shfl_sync(FULL, nl, lb);
        bool on = false;
        uint32_t np = 0, Pk = 0, Nk = 0;
        bool a_many = true;
        if (lane < COUL_NCLS) {
            if (la == lb) {
                on = Na >= 2u && (lane == 0 || P.heavy_step);
                Pk = Na / 2u - (Na % 2u);
                np = Pk + (Na % 2u ? 3u : 0u);
                Nk = Na;
            } else {
                on = Na >= 1u && Nb >= 1u && (lane < 6 || P.heavy_step);
                a_many = Na >= Nb;
                Nk = a_many ? Na : Nb;
                Pk = a_many ? Nb : Na;
                np = Nk;
            }
        }
        const unsigned mact = __ballot_sync(FULL, on);
        if (mact == 0u && !end) continue;
        const unsigned used = __reduce_or_sync(FULL, on ? (1u << la) | (1u << lb) : 0u);
        // the used lists' places in the cache, the classes' first pairs
        uint32_t ncum = (used >> lane) & 1u ? nl : 0u, pcum = on ? np : 0u;
        const uint32_t nown = ncum, pown = pcum;
#pragma unroll
        for (int d = 1; d < 8; d <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, ncum, d);
            if (lane >= d) ncum += y;
        }
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, pcum, d);
            if (lane >= d) pcum += y;
        }
        const uint32_t ctot = __shfl_sync(FULL, ncum, COUL_NLIST - 1), cT = __shfl_sync(FULL, pcum, 31);
        const int r = end ? run : run_of(P, c);
        if (ncl > 0 && (end || r != run || ncl + __popc(mact) > 32 || nlist + __popc(used) > 32 ||
                        tot + ctot > (uint32_t)COUL_CACHE)) {
            const RunInfo* RI = &P.runs[run];
            __syncwarp();
            // the classes' keys
            uint32_t cs = 0xFFFFFFFFu;
            if (lane < ncl) {
                CoulClass& K = W.cl[lane];
                Stream ps(K.lc, step, SID_COUL_PERM | (uint32_t)K.cls, RI->seed, RI->run);
                K.k1 = make_uint4(ps.next(), ps.next(), ps.next(), ps.next());
                if (K.spa != K.spb) K.k2 = make_uint4(ps.next(), ps.next(), ps.next(), ps.next());
                const uint32_t row = RI->row_base + K.lc % (uint32_t)RI->nr;
                const double w = K.cls < 6 ? cw[row] : cw[P.cw_heavy + row];
                K.Kn = (float)(cc.kc[K.cls] * (double)(K.spa == K.spb ? K.N : K.P) * w);
                const bool ei = K.cls >= 1 && K.cls < 6;
                K.fa = ei ? cc.a_e : 0.5f;
                K.fb = ei ? cc.a_t : 0.5f;
                cs = W.start[lane];
            }
            const uint32_t ls = lane < nlist ? W.lcoff[lane] : 0xFFFFFFFFu;
            const uint32_t lo = lane < nlist ? W.lbase[lane] - W.lcoff[lane] : 0u;      // slot of cache place 0
            // which of the batch's classes (lists) an index belongs to: those that
            // start at or before it, of which the first lanes hold the starts in order
            auto owner = [&](uint32_t starts, uint32_t i0) -> int {
                const int before = __popc(__ballot_sync(FULL, starts < i0));
                const uint32_t here = starts - i0 < 32u ? 1u << (starts - i0) : 0u;
                const uint32_t m = __reduce_or_sync(FULL, starts >= i0 ? here : 0u);
                return before + __popc(m & (lt | (1u << lane))) - 1;
            };
            const bool cached = tot <= (uint32_t)COUL_CACHE;
            if (cached)
                for (uint32_t i0 = 0; i0 < tot; i0 += 32) {
                    const uint32_t i = i0 + (uint32_t)lane, slot = __shfl_sync(FULL, lo, owner(ls, i0)) + i;
                    if (i < tot) {
                        cvz[i] = A.vz[slot];
                        cvr[i] = A.vr[slot];
                        cvt[i] = A.vt[slot];
                    }
                }
            for (int k = lane; k < COUL_MASKS; k += 32) mask[k] = 0u;
            __syncwarp();
            float* VZ = cached ? cvz : A.vz;
            float* VR = cached ? cvr : A.vr;
            float* VT = cached ? cvt : A.vt;
#pragma unroll 1
            for (uint32_t c0 = 0; c0 < T; c0 += 32) {
                // lane q: pair c0 + q's particles and draws
                const uint32_t p = c0 + (uint32_t)lane;
                const int j = owner(cs, c0);
                const CoulClass& K = W.cl[j];
                uint32_t ia = 0, ib = 0;
                float z = 0.0f, cph = 1.0f, sph = 0.0f, Kn = 0.0f;
                bool valid = false, fail = false;
                if (p < T) {
                    const uint32_t k = p - W.start[j];
                    uint32_t ra, rb;
                    Kn = K.Kn;
                    if (K.spa == K.spb) {
                        const uint32_t N = K.N;
                        const int h = perm_bits(N);
                        uint32_t xa = 2u * k, xb = 2u * k + 1u;
                        if (k >= K.P) {              // the closing triple: pair q joins q and q + 1 (mod 3)
                            const uint32_t q = k - K.P;
                            xa = N - 3u + q;
                            xb = N - 3u + (q + 1u) % 3u;
                            Kn = Kn * 0.5f;
                        }
                        perm_index2(xa, N, K.k1, h, xb, N, K.k1, h, ra, rb);
                    } else {
                        uint32_t m, f;
                        perm_index2(k, K.N, K.k1, perm_bits(K.N), k % K.P, K.P, K.k2, perm_bits(K.P), m, f);
                        ra = K.flags & 1u ? m : f;
                        rb = K.flags & 1u ? f : m;
                    }
                    const uint32_t pa = K.flags & 2u ? ra : S.table[K.ba + ra];
                    const uint32_t pb = K.flags & 4u ? rb : S.table[K.bb + rb];
                    // the draws do not depend on the particles: they are computed
                    // while the rank lookups are in flight (and dropped for a pair
                    // that does not take place)
                    coul_draws(K.lc, step, sid_coul(K.cls, k), RI->seed, RI->run, z, cph, sph, fail);
                    if (pa < K.na && pb < K.nb) {
                        const uint32_t ka = A.key[K.ba + pa], kb = A.key[K.bb + pb];
                        valid = !(ka & KEY_FLAG) && key_species(ka) == K.spa && !(kb & KEY_FLAG) &&
                                key_species(kb) == K.spb;
                        ia = (cached ? K.ca : K.ba) + pa;
                        ib = (cached ? K.cb : K.bb) + pb;
                    } else {
                        set_error(st, ERR_BOUNDS);   // ids not unique: corrupt state, never index with it
                    }
                }
                const float fa = K.fa, fb = K.fb;
                const int cls = K.cls;
                uint32_t* const ma = mask + ia % COUL_MASKS;
                uint32_t* const mb = mask + ib % COUL_MASKS;
                if (valid) {
                    atomicOr(ma, 1u << lane);
                    atomicOr(mb, 1u << lane);
                }
                __syncwarp();
                uint32_t wait = (*ma | *mb) & lt;
                if (!cached) {
                    // full words: the lanes that another's bits name, compared one by one
                    uint32_t same = 0;
                    for (unsigned named = __reduce_or_sync(FULL, valid ? wait : 0u); named; named &= named - 1u) {
                        const int q = __ffs((int)named) - 1;
                        const uint32_t qa = __shfl_sync(FULL, ia, q), qb = __shfl_sync(FULL, ib, q);
                        if (qa == ia || qa == ib || qb == ia || qb == ib) same |= 1u << q;
                    }
                    wait &= same;
                }
                __syncwarp();
                if (valid) *ma = *mb = 0u;
                unsigned todo = __ballot_sync(FULL, valid);
#pragma unroll 1
                while (todo) {
                    const bool now = (todo >> lane & 1u) && !(wait & todo);
                    if (now) {
                        V3 va{VZ[ia], VR[ia], VT[ia]}, vb{VZ[ib], VR[ib], VT[ib]};
                        if (coulomb_turn(va, vb, Kn, fa, fb, z, cph, sph)) {
                            VZ[ia] = va.x; VR[ia] = va.y; VT[ia] = va.z;
                            VZ[ib] = vb.x; VR[ib] = vb.y; VT[ib] = vb.z;
                            if (cls == 0) ++n_ee;
                            else if (cls < 6) ++n_ei;
                            else ++n_ii;
                            if (fail) ++n_fb;
                        }
                    }
                    __syncwarp();
                    todo &= ~__ballot_sync(FULL, now);
                }
            }
            if (cached) {
                // the velocities back to their slots
                __syncwarp();
                for (uint32_t i0 = 0; i0 < tot; i0 += 32) {
                    const uint32_t i = i0 + (uint32_t)lane, slot = __shfl_sync(FULL, lo, owner(ls, i0)) + i;
                    if (i < tot) {
                        A.vz[slot] = cvz[i];
                        A.vr[slot] = cvr[i];
                        A.vt[slot] = cvt[i];
                    }
                }
            }
            __syncwarp();
            if (end || r != run) {
                const uint32_t ee = __reduce_add_sync(FULL, n_ee), ei = __reduce_add_sync(FULL, n_ei);
                const uint32_t ii = __reduce_add_sync(FULL, n_ii), fb = __reduce_add_sync(FULL, n_fb);
                n_ee = n_ei = n_ii = n_fb = 0;
                if (lane == 0) {
                    RunState& rsv = P.rs[run];
                    if (ee) atomicAdd(&rsv.ctr[C_COUL_EE], (unsigned long long)ee);
                    if (ei) atomicAdd(&rsv.ctr[C_COUL_EI], (unsigned long long)ei);
                    if (ii) atomicAdd(&rsv.ctr[C_COUL_II], (unsigned long long)ii);
                    if (fb) atomicAdd(&rsv.ctr[C_ISOFB], (unsigned long long)fb);
                }
            }
            ncl = nlist = 0;
            tot = T = 0;
        }
        if (end) break;
        run = r;
        // the cell joins the batch: rank tables of the lists its classes use, then the entries
        const RunInfo* RI = &P.runs[r];
        const uint32_t idn = P.rs[r].id_next;
        const int id_top = idn > 1u ? 31 - __clz((int)(idn - 1u)) : 0;
        uint32_t sorted = 0;
        for (unsigned u = used; u; u &= u - 1u) {
            const int l = __ffs((int)u) - 1;
            const uint32_t n = __shfl_sync(FULL, nl, l), b = __shfl_sync(FULL, bl, l);
            IdList L;
            load_ids(L, A.id, b, n, n, S, sbuf, S.table + b, id_top, true);
            if (L.sorted) sorted |= 1u << l;
        }
        const uint32_t coff = tot + ncum - nown;
        const uint32_t ba = __shfl_sync(FULL, bl, la), bb = __shfl_sync(FULL, bl, lb);
        const uint32_t ca = __shfl_sync(FULL, coff, la), cb = __shfl_sync(FULL, coff, lb);
        if (on) {
            const int e = ncl + __popc(mact & lt);
            CoulClass& K = W.cl[e];
            K.P = Pk;
            K.N = Nk;
            K.lc = c - RI->cell_base;
            K.ba = ba;
            K.na = Na;
            K.ca = ca;
            K.bb = bb;
            K.nb = Nb;
            K.cb = cb;
            K.cls = (uint8_t)lane;
            K.spa = (uint8_t)list_species(la);
            K.spb = (uint8_t)list_species(lb);
            K.flags = (uint8_t)((a_many ? 1u : 0u) | ((sorted >> la) & 1u) << 1 | ((sorted >> lb) & 1u) << 2);
            W.start[e] = T + pcum - pown;
        }
        if ((used >> lane) & 1u) {
            const int e = nlist + __popc(used & lt);
            W.lbase[e] = bl;
            W.lcoff[e] = coff;
        }
        ncl += __popc(mact);
        nlist += __popc(used);
        tot += ctot;
        T += cT;
    }
}

// position of the rank-th smallest id for each lane's rank (lanes with has)
__device__ __forceinline__ uint32_t lookup_ranks(const IdList& L, uint32_t rank, bool has, uint32_t nb, uint32_t* cnt,
                                                 int lane) {
    if (L.sorted) return rank;
    if (L.table) return has ? L.table[rank] : 0u;
    uint32_t pos = 0;
#pragma unroll 1
    for (uint32_t q = 0; q < nb; ++q) {
        const uint32_t p = select8(L.base, L.n, __shfl_sync(FULL, rank, (int)q), L.top, cnt, lane);
        if ((uint32_t)lane == q) pos = p;
    }
    return pos;
}

// One warp per active cell, or a block per cell of BIG_CELL candidates or more.
// What bounds it is neither memory nor arithmetic but the instruction caches, the
// latency of a cell's dependent loads and the largest cell.  Unrolled over the
// classes, with the rank code and the kinematics inlined at every use and the
// accepted candidates applied one by one on lane 0, the kernel was 132 KB long and
// waited for instructions half of the time.  Now each part has one copy
// (rank_list, select8 and the Philox rounds out of line, one loop over the classes,
// one over the candidates to apply; no spills to speak of: at 96 registers and five
// blocks an SM it is slower), and the candidates of a batch are applied in rounds.
// 256 x 512 cells, 4e5 candidates in 1.2e5 cells, the largest with 1300: 2290 ->
// 920 us with one copy of each part, 541 us with the large cells on blocks, then
// evenly spread over the SMs (at 38 % of the issue slots, 16 warps an SM).  Plume
// of 2e7 particles: 214 -> 145 us.
template <bool EXT>
__global__ void __launch_bounds__(32 * COLL_WARPS, 4) k_collide(
    Particles A, RankScratch S, const uint32_t* __restrict__ off, const uint32_t* __restrict__ cnt,
    const uint4* __restrict__ nc, const uint4* __restrict__ nc2, const uint32_t* __restrict__ cand_off,
    const uint32_t* __restrict__ active, DevState* st, long long* rho_e, long long* rho_h,
    const float* __restrict__ xsE, const float* __restrict__ xs, KParams P, CollConsts cc, uint32_t big_blocks) {
    if (block_faulted(st)) return;                   // a fault was flagged: the state is not stepped further
    __shared__ __align__(16) uint32_t s_sort[COLL_WARPS][COLL_SORT_WORDS + 2 * RANK_WARP_MAX];
    __shared__ uint32_t s_ctr[COLL_WARPS][OUT_N];
    __shared__ uint32_t s_nsp[COLL_WARPS];           // electrons each warp of a block's batch made
    __shared__ int s_how[2];                         // how the cell's lists are ranked (rank_list by warp 0)
    const int lane = threadIdx.x & 31, wib = (threadIdx.x >> 5) & (COLL_WARPS - 1);
    uint32_t* ctr = s_ctr[wib];
    if (lane < OUT_N) ctr[lane] = 0u;
    __syncwarp();
    const uint32_t C = P.ncell;
    const uint32_t n_heavy = st->n_heavy, n_light = st->n_light;
    const uint32_t n_alive = (uint32_t)st->tail_base;   // spawn slots follow the bins
    // a counter's place in RunState::ctr
    auto flush = [&](int r) {
        __syncwarp();
        if (lane < OUT_N && ctr[lane]) {
            const int c = lane < NCH ? c_event(lane) : lane == OUT_NULL ? C_NULL : lane == OUT_CONSUMED ? C_CONSUMED
                        : lane == OUT_THR ? C_THR : lane == OUT_VIOL ? C_VIOL : C_ISOFB;
            atomicAdd(&P.rs[r].ctr[c], (unsigned long long)ctr[lane]);
            ctr[lane] = 0u;
        }
        __syncwarp();
    };
    // The big cells first, a block each: the first blocks (those resident from
    // the start) look for them among the heavy ones.  Then the other heavy cells,
    // taken one at a time from a shared cursor by the first min(n_heavy, warps)
    // warps, and the light cells, warp-strided.
    const uint32_t warp0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    bool heavy_phase = warp0 < n_heavy;
    uint32_t wl = warp0, wb = blockIdx.x < big_blocks ? blockIdx.x : n_heavy;
    uint32_t tag = 0;                                // rounds of the block so far
    for (;;) {
        bool blk = false;                            // (the same in all warps of the block while there are big cells)
        uint32_t c = 0;
        while (wb < n_heavy && !blk) {
            c = active[wb];
            wb += big_blocks;
            blk = (c & BIG_FLAG) != 0u;
        }
        c &= ~BIG_FLAG;
        if (!blk && heavy_phase) {
            uint32_t w = 0;
            if (lane == 0) w = atomicAdd(&st->collide_next, 1u);
            w = __shfl_sync(FULL, w, 0);
            if (w < n_heavy) {
                c = active[w];
                if (c & BIG_FLAG) continue;
            } else {
                heavy_phase = false;
            }
        }
        if (!blk && !heavy_phase) {
            if (wl >= n_light) break;
            c = active[C - 1u - wl];
            wl += nwarps;
        }
        // the group that takes the cell: this warp, or the block (with warp 0's buffers)
        const uint32_t GS = blk ? 32u * COLL_WARPS : 32u, me = blk ? threadIdx.x : (uint32_t)lane;
        uint32_t* sbuf = s_sort[blk ? 0 : wib];          // rank_list's buffers and counters,
        uint32_t* tab0 = sbuf + COLL_SORT_WORDS;         // then the tables of the pair's two lists
        auto ranks = [&](IdList& L, int which, uint32_t slot0, uint32_t n, uint32_t lookups, int id_top) {
            if (!blk) {
                load_ids(L, A.id, slot0, n, lookups, S, sbuf, tab0 + which * RANK_WARP_MAX, id_top);
                return;
            }
            __syncthreads();                             // the buffers' last readers are done
            if (wib == 0) {
                load_ids(L, A.id, slot0, n, lookups, S, sbuf, tab0 + which * RANK_WARP_MAX, id_top);
                if (lane == 0) s_how[which] = L.sorted ? 0 : L.table ? 1 : 2;
            }
            __syncthreads();
            const int how = s_how[which];
            L.n = n;
            L.base = A.id + slot0;
            L.top = id_top;
            L.sorted = how == 0;
            L.table = how == 1 ? (n > 32u * RC ? S.table + slot0 : tab0 + which * RANK_WARP_MAX) : nullptr;
        };
        const uint4 n = nc[c];         // candidates of the classes (e,Cu), (e,Cu+), (Cu,Cu+), (Cu,Cu)
        // and of (e,Cu2+ SW), (e,Cu2+ DI), (e,Cu3+)
        const uint4 n2 = EXT && P.charge_max >= 3 ? nc2[c] : make_uint4(0u, 0u, 0u, 0u);
        const uint32_t e_base = off[c], Ne = cnt[c], co = cand_off[c];
        const int r = run_of(P, c);
        const RunInfo* RI = &P.runs[r];
        const uint32_t lc = c - RI->cell_base;
        const uint32_t nres = 2u * (n.x + n.y + n2.x + n2.y + n2.z);     // reserved spawn slots
        const unsigned long long slot0 = (unsigned long long)n_alive + 2ull * co;
        // ids: the run's next id plus twice the candidates of the run's earlier
        // cells; every id in the cell's lists is below the run's next id
        const uint32_t idn = P.rs[r].id_next;
        const uint32_t id0 = idn + 2u * (co - cand_off[RI->cell_base]);
        const int id_top = idn > 1u ? 31 - __clz((int)(idn - 1u)) : 0;
        uint32_t nspawn = 0;
        if (slot0 + nres > P.capacity) {
            // no room for this cell's spawns: report, and leave its reserved
            // slots (those that exist) dead
            if (me == 0) set_error(st, ERR_CAPACITY);
#pragma unroll 1
            for (unsigned long long q = slot0 + me; q < P.capacity && q < slot0 + nres; q += GS) A.key[q] = DEAD;
            continue;
        }
        // lookups of each list over all classes (the rank-table decisions of
        // k_ncand use the same totals): the Coulomb pairs look up every
        // electron and every ion of a cell with electrons
        // (ion pairs collide on heavy steps even where there are no electrons)
        const bool coul_e = EXT && P.coulomb && Ne > 0;
        const bool coul = EXT && P.coulomb && (Ne > 0 || P.heavy_step);
        const uint32_t look_e = n.x + n.y + n2.x + n2.y + n2.z + (coul_e ? Ne : 0u);
        const uint32_t look_cu = n.x + n.z + 2u * n.w, look_ci = n.y + n.z;
        // the first list of a pair: electrons for the electron classes, Cu for
        // the heavy classes (loaded over the electrons' list once those are done)
        IdList el;
        uint32_t a_base = e_base, Na = Ne;
        bool cu_first = false;
        if (look_e) ranks(el, 0, e_base, Ne, look_e, id_top);
#pragma unroll 1
        for (int k = 0; k < (EXT ? NCLS : 2); ++k) {
            const uint32_t ncand = k == 0 ? n.x : k == 1 ? n.y : k == 2 ? n2.x : k == 3 ? n2.y : k == 4 ? n2.z
                                 : k == 5 ? n.z : n.w;
            if (ncand == 0) continue;
            if (EXT && k >= NECLS && !cu_first) {
                cu_first = true;
                a_base = off[C + c];
                Na = cnt[C + c];
                ranks(el, 0, a_base, Na, look_cu, id_top);
            }
            const int ts = class_target(k);
            const uint32_t tb = (uint32_t)ts * C + c;
            const uint32_t t_base = off[tb];
            const uint32_t Nt = cnt[tb];
            // the target list's lookups over every class that draws from it
            const uint32_t t_look = ts == SP_CU ? look_cu : (ts == SP_CUP ? look_ci : ncand) + (coul ? Nt : 0u);
            IdList tl;
            ranks(tl, 1, t_base, Nt, t_look, id_top);
            // candidates in batches: thread q of the group draws candidate m0 + q's pair
#pragma unroll 1
            for (uint32_t m0 = 0; m0 < ncand; m0 += GS) {
                const uint32_t nb = min(GS, ncand - m0);
                const bool has = me < nb;
                uint32_t i = 0, j = 0;
                float Racc = 0.0f, Rch = 0.0f;
                if (has) {
                    const uint4 d = philox_block(make_uint4(lc, st->step, sid_cand(k, m0 + me), 0u),
                                                 make_uint2(RI->seed, RI->run));
                    i = (uint32_t)(((unsigned long long)d.x * Na) >> 32);
                    if (EXT && k == 6) {    // a second, different Cu
                        j = (uint32_t)(((unsigned long long)d.y * (Na - 1u)) >> 32);
                        if (j >= i) ++j;
                    } else {
                        j = (uint32_t)(((unsigned long long)d.y * Nt) >> 32);
                    }
                    Racc = __fmul_rn((float)(d.z >> 8), 5.9604644775390625e-08f);
                    Rch = __fmul_rn((float)(d.w >> 8), 5.9604644775390625e-08f);
                }
                // (a select works on its own warp's candidates and counters)
                const uint32_t nw = blk ? (nb > 32u * wib ? min(32u, nb - 32u * wib) : 0u) : nb;
                uint32_t* scnt = s_sort[wib] + 4 * RANK_WARP_MAX;
                const uint32_t pe = lookup_ranks(el, i, has, nw, scnt, lane);
                const uint32_t pt = lookup_ranks(tl, j, has, nw, scnt, lane);
                const bool ok = has && pe < Na && pt < Nt;   // ids not unique: corrupt state, never index with it
                if (has && !ok) set_error(st, ERR_BOUNDS);
                const uint32_t ie = a_base + (ok ? pe : 0u), it = t_base + (ok ? pt : 0u);
                // Applied in rounds: every candidate to apply yet whose earlier
                // sharers of a particle are all through (no two of a round touch
                // the same particle), so that each sees its particles as the
                // sequence leaves them.  A warp compares all pairs of its batch
                // once; a block lets its candidates claim their particles' places
                // in two tables each round, the earliest first (two particles
                // of one place only wait needlessly).  The two particles of a
                // (Cu, Cu) pair come from one list.
                uint32_t conf = 0;
                const uint32_t he = ie & (CLAIMS - 1u), ht = it & (CLAIMS - 1u);
                uint32_t* te = s_sort[1];
                uint32_t* tt = EXT && k == 6 ? te : s_sort[2];
                if (!blk) {
#pragma unroll 1
                    for (uint32_t q = 0; q + 1 < nb; ++q) {
                        const uint32_t e2 = __shfl_sync(FULL, ie, (int)q), t2 = __shfl_sync(FULL, it, (int)q);
                        if (q < (uint32_t)lane && (e2 == ie || t2 == it || (EXT && k == 6 && (e2 == it || t2 == ie))))
                            conf |= 1u << q;
                    }
                } else if (tag == 0u) {
                    for (uint32_t q = me; q < CLAIMS; q += GS) s_sort[1][q] = s_sort[2][q] = 0u;
                    __syncthreads();
                }
                bool pend = ok;
                int out = -1, nsp = 0;
                bool viol = false;
                uint32_t fb = 0;
                Spawn sp[2];
                for (;;) {
                    bool ready;
                    if (!blk) {
                        const uint32_t b = __ballot_sync(FULL, pend);
                        if (!b) break;
                        ready = pend && !(conf & b);
                    } else {
                        // claims of later rounds are larger, of earlier candidates too
                        ++tag;
                        const uint32_t v = tag * (32u * COLL_WARPS) + (32u * COLL_WARPS - 1u - me);
                        if (pend) {
                            atomicMax(&te[he], v);
                            atomicMax(&tt[ht], v);
                        }
                        if (!__syncthreads_or(pend)) break;
                        ready = pend && te[he] == v && tt[ht] == v;
                    }
                    if (ready) {
                        out = collide_pair<EXT>(A, k, ie, it, lc, m0 + me, Racc, Rch, RI, P.geom, xsE, xs, cc, st,
                                                rho_h, viol, fb, nsp, sp);
                        pend = false;
                    }
                    if (blk) __syncthreads();
                    else __syncwarp();
                }
                if (out >= 0) atomicAdd(&ctr[out], 1u);
                if (viol) atomicAdd(&ctr[OUT_VIOL], 1u);
                if (fb) atomicAdd(&ctr[OUT_FB], fb);
                // the electrons made, in candidate order
                const uint32_t b1 = __ballot_sync(FULL, nsp > 0), b2 = __ballot_sync(FULL, nsp > 1);
                uint32_t made = __popc(b1) + __popc(b2), s0 = nspawn;
                if (blk) {
                    if (lane == 0) s_nsp[wib] = made;
                    __syncthreads();
                    made = 0;
#pragma unroll
                    for (int w = 0; w < COLL_WARPS; ++w) {
                        if (w < wib) s0 += s_nsp[w];
                        made += s_nsp[w];
                    }
                }
                nspawn += made;
                if (b1) {
                    const uint32_t lt = (1u << lane) - 1u;
                    s0 += __popc(b1 & lt) + __popc(b2 & lt);
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        if (q >= nsp) continue;
                        if (s0 + q >= nres) {
                            set_error(st, ERR_BOUNDS);
                            continue;
                        }
                        const unsigned long long slot = slot0 + s0 + q;
                        A.key[slot] = make_key(SP_E, sp[q].cell);
                        A.pz[slot] = sp[q].pz;
                        A.pr[slot] = sp[q].pr;
                        A.vz[slot] = sp[q].v.x;
                        A.vr[slot] = sp[q].v.y;
                        A.vt[slot] = sp[q].v.z;
                        A.id[slot] = id0 + s0 + q;
                        deposit1(rho_e, *RI, P.geom, sp[q].cell - RI->cell_base, sp[q].pz, sp[q].pr, -1);
                    }
                }
            }
        }
#pragma unroll 1
        for (uint32_t q = nspawn + me; q < nres; q += GS) A.key[slot0 + q] = DEAD;
        if (P.nruns > 1) flush(r);
    }
    if (P.nruns == 1) flush(0);
}

// slot / id bookkeeping of the step and the RC circuit of each run
__global__ void k_finalize(const uint32_t* __restrict__ off, uint32_t nbins, const uint32_t* __restrict__ cand_off,
                           DevState* st, KParams P, const RunCircuit* __restrict__ circ, double dt, int circuit) {
    const uint32_t C = P.ncell;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const unsigned long long T = cand_off[C];
        unsigned long long ns = st->tail_base + 2ull * T;
        if (ns > P.capacity) {
            set_error(st, ERR_CAPACITY);
            ns = P.capacity;
        }
        // the next step's particles (in bins and in the spawn slots) within
        // the configured capacity
        if (st->n_live + st->n_e + 2ull * T > P.user_capacity) set_error(st, ERR_CAPACITY);
        st->n_slots = ns;
        st->n_bigc = 0;
        st->n_ovf = 0;
        st->since += 1u;
        st->n_heavy = 0;
        st->n_light = 0;
        st->n_mid = 0;
        st->n_big = 0;
        st->collide_next = 0;
        st->n_sput = 0;
    }
    // the step is over for every kernel that draws from it
    if (blockIdx.x == 0 && threadIdx.x == 0) st->step += 1u;
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < P.nruns; r += gridDim.x * blockDim.x) {
        const RunInfo& RI = P.runs[r];
        RunState& rs = P.rs[r];
        const unsigned long long T = cand_off[RI.cell_base + RI.ncell] - cand_off[RI.cell_base];
        if ((unsigned long long)rs.id_next + 2ull * T > 0xFFFFFFFFull) set_error(st, ERR_IDS);
        rs.id_next += (uint32_t)(2ull * T);
        rs.ctr[C_CAND] += T;
        if (circuit) {
            // C dV/dt = (V0 - V)/R - I_gap; the gap current leaves the anode node
            const double I = -rs.anode_charge_step / dt;
            rs.I_gap = I;
            rs.V += dt / circ[r].C_farad * ((circ[r].V0 - rs.V) / circ[r].R_ohm - I);
            rs.anode_charge_step = 0.0;
        }
    }
}

// ---------------------------------------------------------------------
// cathode injection (Sec. 2.3): FN electrons from the tip and neutrals at
// a fixed fraction of the electron flux; one block per run.
// ---------------------------------------------------------------------
__device__ __forceinline__ float rayleigh(const float* __restrict__ ray, float U) {
    const float x = U * 1023.0f;
    const int k = min((int)x, 1022);
    const float t = x - (float)k;
    return ray[k] + t * (ray[k + 1] - ray[k]);
}

__global__ void __launch_bounds__(256) k_inject(Particles A, const float2* __restrict__ E, DevState* st, KParams P,
                                                const InjectConsts* __restrict__ icv, const float* __restrict__ ray) {
    if (block_faulted(st)) return;                   // a fault was flagged: the state is not stepped further
    __shared__ uint32_t ne_s[64], nn_s[64], pre_s[65];
    __shared__ unsigned long long slot0_s;
    const int run = blockIdx.x;
    const InjectConsts& ic = icv[run];
    const RunInfo& RI = P.runs[run];
    RunState& rs = P.rs[run];
    if (ic.ntip == 0) return;
    const int t = threadIdx.x;
    if (t < ic.ntip) {
        const int j = t;
        const double ezs = 0.5 * ((double)E[node_of(RI, 0, 0, j)].x + (double)E[node_of(RI, 0, 0, j + 1)].x);
        const double F = ic.beta * (ezs < 0 ? -ezs : 0.0);
        double J = 0.0;
        if (F > 0.0) {
            const double Afn = 1.541434e-6, Bfn = 6.830890e9;
            J = Afn / ic.work * F * F * exp(-Bfn * ic.work * sqrt(ic.work) / F);
        }
        const double lam_e = J * ic.area[j] * ic.dt / (1.602176634e-19 * ic.weight);
        const double lam_n = ic.ratio * lam_e;
        Stream s((uint32_t)j, st->step, SID_INJ_COUNT, RI.seed, RI.run);
        const double Re = (double)s.u01(), Rn = (double)s.u01();
        ne_s[j] = (uint32_t)floor(lam_e + Re);
        nn_s[j] = (uint32_t)floor(lam_n + Rn);
    }
    __syncthreads();
    if (t == 0) {
        uint32_t acc = 0;
        for (int j = 0; j < ic.ntip; ++j) {
            pre_s[j] = acc;
            acc += ne_s[j] + nn_s[j];
        }
        pre_s[ic.ntip] = acc;
        slot0_s = acc ? atomicAdd(&st->n_slots, (unsigned long long)acc) : 0ull;
    }
    __syncthreads();
    const uint32_t total = pre_s[ic.ntip];
    const unsigned long long slot0 = slot0_s;
    const uint32_t id0 = rs.id_next;
    uint32_t emitted_e = 0, emitted_cu = 0;
    uint32_t fb = 0;
    for (uint32_t p = t; p < total; p += blockDim.x) {
        int j = 0;
        while (pre_s[j + 1] <= p) ++j;
        const uint32_t loc = p - pre_s[j];
        const bool is_e = loc < ne_s[j];
        Stream sp((uint32_t)j, st->step, is_e ? sid_inj_e(loc) : sid_inj_cu(loc - ne_s[j]), RI.seed, RI.run);
        const float U = sp.u01();
        const float lo = ic.lo[j], hi = ic.hi[j];
        const float rr = sqrtf(lo * lo + U * (hi * hi - lo * lo));
        float pr = rr - lo;
        if (pr >= 1.0f) pr = 0x1.fffffep-1f;
        if (pr < 0.0f) pr = 0.0f;
        float vz = 0.f, vr = 0.f, vt = 0.f;
        if (!is_e) {
            const float U1 = sp.u01(), U2 = sp.u01();
            vz = ic.vth * rayleigh(ray, U1);
            const float s = ic.vth * rayleigh(ray, U2);
            float cp, sn;
            azimuth(sp, cp, sn, fb);
            vr = s * cp;
            vt = s * sn;
        }
        const unsigned long long slot = slot0 + p;
        if (slot >= P.capacity) {
            set_error(st, ERR_CAPACITY);
            continue;
        }
        A.key[slot] = make_key(is_e ? SP_E : SP_CU, RI.cell_base + (uint32_t)j);   // iz = 0
        A.pz[slot] = 0.0f;
        A.pr[slot] = pr;
        A.vz[slot] = vz;
        A.vr[slot] = vr;
        A.vt[slot] = vt;
        A.id[slot] = id0 + p;
        if (is_e) ++emitted_e; else ++emitted_cu;
    }
    if (emitted_e) {
        atomicAdd(&rs.ctr[C_EMIT_E], (unsigned long long)emitted_e);
        for (uint32_t q = 0; q < emitted_e; ++q) atomicAdd(&rs.charge_cathode, 1.602176634e-19 * ic.weight);
    }
    if (emitted_cu) atomicAdd(&rs.ctr[C_EMIT_CU], (unsigned long long)emitted_cu);
    if (fb) atomicAdd(&rs.ctr[C_ISOFB], (unsigned long long)fb);
    __syncthreads();
    if (t == 0) {
        rs.id_next = id0 + total;
        if (slot0 + total > P.capacity) atomicMin(&st->n_slots, P.capacity);
    }
}

constexpr size_t RT_SMEM = (size_t)RANK_BLOCK_MAX * 4 * sizeof(uint32_t);
constexpr size_t RT_MID_SMEM = (size_t)RANK_MID_MAX * 4 * sizeof(uint32_t);

// ---------------------------------------------------------------------
// Ion-impact sputtering (Sec. 2.3), after the push: each run's block takes
// the impacts the push recorded for it, sorts them by the ion's id, and
// appends their atoms after the slots in use, as movers that the sort which
// follows places, with ids from the run's next id in that order.  An atom leaves the
// impact point on the electrode surface with an effusive flux at
// sputter_T: Rayleigh normal and transverse speeds, uniform azimuth.
// ---------------------------------------------------------------------
constexpr int SPUT_THREADS = 1024;
constexpr uint32_t SPUT_MAX = 8192;              // impacts per run and step
constexpr size_t SPUT_SMEM = SPUT_MAX * sizeof(unsigned long long);

__global__ void __launch_bounds__(SPUT_THREADS) k_sputter(Particles M, uint32_t* mm, DevState* st, KParams P,
                                                          const float* __restrict__ ray, uint32_t* in_cnt) {
    if (block_faulted(st)) return;                   // a fault was flagged: the state is not stepped further
    extern __shared__ unsigned long long s_key[];    // ion id << 32 | record index
    __shared__ uint32_t s_cnt, s_el[2], s_wsum[SPUT_THREADS / 32];
    __shared__ unsigned long long s_base;
    __shared__ uint32_t s_id0, s_ok;
    const int r = blockIdx.x;
    const uint32_t tid = threadIdx.x;
    const uint32_t nq = min(st->n_sput, P.squeue_cap);
    if (tid == 0) {
        s_cnt = 0u;
        s_el[0] = s_el[1] = 0u;
    }
    __syncthreads();
    for (uint32_t x = tid; x < nq; x += SPUT_THREADS) {
        const SputRec rec = P.squeue[x];
        if ((int)(rec.meta >> 1) != r) continue;
        const uint32_t k = atomicAdd(&s_cnt, 1u);
        if (k < SPUT_MAX) s_key[k] = ((unsigned long long)rec.id << 32) | x;
    }
    __syncthreads();
    const uint32_t m = s_cnt;
    if (m == 0u) return;
    if (m > SPUT_MAX) {
        if (tid == 0) set_error(st, ERR_CAPACITY);
        return;
    }
    // bitonic sort of the keys, padded with all-ones to a power of two
    uint32_t np2 = 1u;
    while (np2 < m) np2 <<= 1;
    for (uint32_t x = m + tid; x < np2; x += SPUT_THREADS) s_key[x] = ~0ull;
    __syncthreads();
    for (uint32_t kk = 2u; kk <= np2; kk <<= 1)
        for (uint32_t j = kk >> 1; j > 0u; j >>= 1) {
            for (uint32_t x = tid; x < np2; x += SPUT_THREADS) {
                const uint32_t y = x ^ j;
                if (y > x) {
                    const unsigned long long a = s_key[x], b = s_key[y];
                    if ((a > b) == ((x & kk) == 0u)) {
                        s_key[x] = b;
                        s_key[y] = a;
                    }
                }
            }
            __syncthreads();
        }
    // atoms per impact in id order: each thread a contiguous chunk, an
    // exclusive scan of the chunk sums across the block
    const uint32_t per = (m + SPUT_THREADS - 1u) / SPUT_THREADS;
    const uint32_t c0 = min(tid * per, m), c1 = min(c0 + per, m);
    uint32_t sum = 0;
    for (uint32_t i = c0; i < c1; ++i) {
        const SputRec rec = P.squeue[(uint32_t)s_key[i]];
        sum += rec.n;
        atomicAdd(&s_el[rec.meta & 1u], rec.n);
    }
    const int lane = (int)(tid & 31u), w = (int)(tid >> 5);
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) s_wsum[w] = incl;
    __syncthreads();
    if (w == 0) {
        uint32_t v = s_wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(FULL, v, o);
            if (lane >= o) v += u;
        }
        s_wsum[lane] = v;                            // inclusive warp totals
    }
    __syncthreads();
    const uint32_t total = s_wsum[SPUT_THREADS / 32 - 1];
    uint32_t off = (w > 0 ? s_wsum[w - 1] : 0u) + incl - sum;
    if (tid == 0) {
        const unsigned long long base = atomicAdd(&st->n_slots, (unsigned long long)total);
        s_ok = base + total <= P.capacity ? 1u : 0u;
        if (!s_ok) set_error(st, ERR_CAPACITY);
        s_base = base;
        RunState& rs = P.rs[r];
        s_id0 = rs.id_next;
        if ((unsigned long long)rs.id_next + total > 0xFFFFFFFFull) set_error(st, ERR_IDS);
        rs.id_next += total;
        if (s_el[0]) rs.ctr[C_SPUT_C] += s_el[0];
        if (s_el[1]) rs.ctr[C_SPUT_A] += s_el[1];
    }
    __syncthreads();
    if (!s_ok) return;
    const RunInfo& RI = P.runs[r];
    uint32_t fb = 0;
    for (uint32_t i = c0; i < c1; ++i) {
        const SputRec rec = P.squeue[(uint32_t)s_key[i]];
        const uint32_t el = rec.meta & 1u;
        const int iz = el == 0u ? 0 : RI.nz - 1;
        const float pz = el == 0u ? 0.0f : 0x1.fffffep-1f;
        const uint32_t gcell = RI.cell_base + (uint32_t)iz * (uint32_t)RI.nr + rec.ir;
        for (uint32_t j = 0; j < rec.n; ++j, ++off) {
            Stream sp(rec.id, st->step, sid_sput_atom(j), RI.seed, RI.run);
            const float U1 = sp.u01(), U2 = sp.u01();
            const float vn = P.sput_vth * rayleigh(ray, U1);
            const float sv = P.sput_vth * rayleigh(ray, U2);
            float cp, sn;
            azimuth(sp, cp, sn, fb);
            // a tail slot after those in use: the atom joins this step's sort as a mover
            const unsigned long long slot = s_base + off;
            M.key[slot] = make_key(SP_CU, gcell);
            M.pz[slot] = pz;
            M.pr[slot] = rec.pr;
            M.vz[slot] = el == 0u ? vn : -vn;
            M.vr[slot] = sv * cp;
            M.vt[slot] = sv * sn;
            M.id[slot] = s_id0 + off;
            atomicOr(&mm[slot >> 5], 1u << (slot & 31u));
            atomicAdd(&in_cnt[(uint32_t)SP_CU * P.ncell + gcell], 1u);
        }
    }
    if (fb) atomicAdd(&P.rs[r].ctr[C_ISOFB], (unsigned long long)fb);
}

cudaError_t collide_setup() {
    cudaError_t e = cudaFuncSetAttribute(k_rank_tables<RT_THREADS, RANK_BLOCK_MAX>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RT_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_rank_tables<RT_MID_THREADS, RANK_MID_MAX>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RT_MID_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sputter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SPUT_SMEM);
    return e;
}
void launch_ncand(const uint32_t* cnt, const float* ck, uint4* nc, uint4* nc2, uint32_t* cand, uint32_t* active,
                  uint32_t* mid, uint32_t* big, DevState* st, const KParams& P, int grid, cudaStream_t s) {
    if (P.charge_max >= 3 || P.heavy_coll || P.coulomb)
        k_ncand<true><<<grid, 256, 0, s>>>(cnt, ck, nc, nc2, cand, active, mid, big, st, P);
    else
        k_ncand<false><<<grid, 256, 0, s>>>(cnt, ck, nc, nc2, cand, active, mid, big, st, P);
}
void launch_collide(const Particles& A, const Particles& B, const uint32_t* off, const uint32_t* cnt, const uint4* nc,
                    const uint4* nc2,
                    const uint32_t* cand_off, const uint32_t* active, const uint32_t* mid, const uint32_t* big,
                    DevState* st, long long* rho_e, long long* rho_h, const float* xsE, const float* xs,
                    const KParams& P, const CollConsts& cc, int sms, int grid, cudaStream_t s) {
    const RankScratch S{B.key, reinterpret_cast<uint32_t*>(B.pz), reinterpret_cast<uint32_t*>(B.pr),
                        reinterpret_cast<uint32_t*>(B.vz), B.id};
    k_rank_tables<RT_MID_THREADS, RANK_MID_MAX><<<sms * RT_MID_BLOCKS_PER_SM, RT_MID_THREADS, RT_MID_SMEM, s>>>(
        A.id, S, off, cnt, mid, &st->n_mid, rank_queue_max(P.capacity, RANK_WARP_MAX), P.ncell, st);
    k_rank_tables<RT_THREADS, RANK_BLOCK_MAX><<<sms, RT_THREADS, RT_SMEM, s>>>(
        A.id, S, off, cnt, big, &st->n_big, rank_queue_max(P.capacity, RANK_MID_MAX), P.ncell, st);
    const uint32_t nbig = (uint32_t)std::min(grid, 4 * sms);      // blocks resident from the start
    if (P.charge_max >= 3 || P.heavy_coll || P.coulomb)
        k_collide<true><<<grid, 32 * COLL_WARPS, 0, s>>>(A, S, off, cnt, nc, nc2, cand_off, active, st, rho_e, rho_h,
                                                         xsE, xs, P, cc, nbig);
    else
        k_collide<false><<<grid, 32 * COLL_WARPS, 0, s>>>(A, S, off, cnt, nc, nc2, cand_off, active, st, rho_e, rho_h,
                                                          xsE, xs, P, cc, nbig);
}
void launch_coulomb(const Particles& A, const Particles& B, const uint32_t* off, const uint32_t* cnt, DevState* st,
                    const KParams& P, const CollConsts& cc, const double* cw, int sms, cudaStream_t s) {
    const RankScratch S{B.key, reinterpret_cast<uint32_t*>(B.pz), reinterpret_cast<uint32_t*>(B.pr),
                        reinterpret_cast<uint32_t*>(B.vz), B.id};
    // a full batch a warp; fewer cells where that would leave the SMs short of warps
    // (four steps of 97 x 131 cells 2.17 -> 1.80 ms, of 41 x 43 cells 1.05 -> 0.80)
    const uint32_t cells = std::min<uint32_t>(std::max<uint32_t>(P.ncell / (uint32_t)(sms * COUL_BLOCKS), 1u), COUL_CELLS);
    k_coulomb<<<(P.ncell + cells - 1) / cells, 32, 0, s>>>(A, S, off, cnt, st, P, cc, cw, cells);
}
void launch_finalize(const uint32_t* off, uint32_t nbins, const uint32_t* cand_off, DevState* st, const KParams& P,
                     const RunCircuit* circ, double dt, int circuit, cudaStream_t s) {
    k_finalize<<<1, 256, 0, s>>>(off, nbins, cand_off, st, P, circ, dt, circuit);
}
void launch_sputter(const Particles& M, uint32_t* mm, DevState* st, const KParams& P, const float* ray,
                    uint32_t* in_cnt, cudaStream_t s) {
    k_sputter<<<P.nruns, SPUT_THREADS, SPUT_SMEM, s>>>(M, mm, st, P, ray, in_cnt);
}

void launch_inject(Particles A, const float2* E, DevState* st, const KParams& P, const InjectConsts* ic,
                   const float* ray, cudaStream_t s) {
    k_inject<<<P.nruns, 256, 0, s>>>(A, E, st, P, ic, ray);
}

}  // namespace pd
