// pd_warp.cuh -- warp-level aggregation helpers shared by the particle kernels.
#pragma once
#include "pd_internal.cuh"

namespace pd {

constexpr unsigned FULL_MASK = 0xFFFFFFFFu;

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ long long warp_sum_ll(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
    return v;
}
__device__ __forceinline__ unsigned long long warp_sum_ull(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
    return v;
}

// Fixed-point CIC deposit, Eq. (9)-(10): w = rn(f * 2^16) per axis, corner
// weights (2^16 - w_z)(2^16 - w_r), w_z (2^16 - w_r), (2^16 - w_z) w_r, w_z w_r
// (they sum to 2^32).  Lanes holding the same key (species and cell) are
// summed first: the four corners follow from the sums of w_z, w_r and their
// product, the product in 16-bit halves so that the warp sums fit in 32 bits;
// then one 64-bit atomic per node and group.  rho and zq may differ between keys.
__device__ __forceinline__ void warp_deposit(long long* rho, const RunInfo& RI, int geom, uint32_t key, float pz,
                                             float pr, int zq, bool on) {
    const unsigned m = __ballot_sync(FULL_MASK, on);
    if (!on) return;
    const unsigned g = __match_any_sync(m, key);
    const uint32_t wz = __float2uint_rn(pz * 65536.0f);
    const uint32_t wr = __float2uint_rn(pr * 65536.0f);
    const unsigned long long w = (unsigned long long)wz * wr;
    const uint32_t sz = __reduce_add_sync(g, wz), sr = __reduce_add_sync(g, wr);
    const uint32_t hi = __reduce_add_sync(g, (uint32_t)(w >> 16)), lo = __reduce_add_sync(g, (uint32_t)w & 0xFFFFu);
    if ((threadIdx.x & 31) == (unsigned)(__ffs(g) - 1)) {
        const uint32_t lc = key_cell(key) - RI.cell_base, nr = (uint32_t)RI.nr;
        const int iz = (int)(lc / nr), ir = (int)(lc - (uint32_t)iz * nr);
        const long long zr = ((long long)hi << 16) + lo, z0 = ((long long)sz << 16) - zr, r0 = ((long long)sr << 16) - zr;
        const long long q = ((long long)__popc(g) << 32) - z0 - r0 - zr;
        auto add = [&](int i, int j, long long v) {
            atomicAdd((unsigned long long*)&rho[node_of(RI, geom, i, j)], (unsigned long long)(v * zq));
        };
        add(iz, ir, q);
        add(iz + 1, ir, z0);
        add(iz, ir + 1, r0);
        add(iz + 1, ir + 1, zr);
    }
}

}  // namespace pd
