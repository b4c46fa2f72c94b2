// pd_net.cu -- the network of the learned Poisson warm start: inference,
// back-propagation of the mean squared error and Adam, all on the GPU.
//
// Six 3 x 3 convolutions over node grids (zero padding), channels 1 -> 32 ->
// 32 -> 32 -> 32 -> 32 -> 1, ReLU after the first five.  The four 32 -> 32
// layers, forward and back-propagation alike, are implicit GEMMs on the
// tensor cores (mma.sync m16n8k16, bfloat16 operands, float accumulators):
//   forward / input gradient: M = 16 nodes of a tile row, N = 32 output
//     channels, K = 9 taps x 32 input channels; a warp keeps the weights of its
//     16 output channels in registers, a block stages 8 x 32 node tiles with
//     their halo in shared memory.  The input gradient is the same convolution
//     over the output gradient with the weights mirrored in the tap and
//     transposed in the channels.
//   weight gradient: per tap, M = 32 output channels, N = 32 input channels,
//     K = the nodes, with one warp per tap; each block sums over the tiles it
//     visits and writes a partial that a second kernel adds up in a fixed
//     order (so the gradient does not depend on the launch).
// The 1 -> 32 layer, and the 32 -> 1 layer in training, run on the CUDA cores (the
// latter in inference on the tensor cores: k_conv6).
// Storage: activations h_1..h_5 and the gradients with respect to a_1..a_5 in
// bfloat16 (node-major, 32 channels = 64 bytes per node), the input, output,
// targets and the output gradient in float, weights in bfloat16 for the layers and
// in float (master copies) for Adam.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "pd.h"
#include "pd_launch.cuh"
#include "pd_net.h"

namespace pd {
namespace {

using bf16 = __nv_bfloat16;
constexpr int CH = 32;
constexpr int NP = PD_NET_NPARAMS;
// offsets of layer l's weights and biases in the parameter vector (layer 0:
// 288 weights + 32 biases; layers 1-4: 9216 + 32; layer 5: 288 + 1)
__host__ __device__ constexpr int off_w(int l) { return l == 0 ? 0 : (l < 5 ? 320 + (l - 1) * 9248 : 37312); }
__host__ __device__ constexpr int off_b(int l) { return l == 0 ? 288 : off_w(l) + (l < 5 ? 9216 : 288); }
static_assert(off_b(5) + 1 == PD_NET_NPARAMS, "parameter layout");
constexpr int TY = 8, TX = 16;       // node tile of the weight gradients
constexpr int CX = 32;               // columns of a convolution's tile (of TY rows)
constexpr int CONV_THREADS = 128;    // a 32 -> 32 layer's block: two column groups by two channel halves
constexpr int HP = 40;               // channel stride of a staged node (bf16): 80 bytes, conflict-free fragments
constexpr int MAX_PART_BLOCKS = 384;  // (k_reduce holds a value's partials in 48 KB of shared memory, 32 values a block)
constexpr int PART_STRIDE = (NP + 31) / 32 * 32;   // a block's partial gradient: the whole parameter vector
constexpr int LOSS_BLOCKS = 256;

size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

__device__ __forceinline__ int tap_dy(int tap) { return tap / 3 - 1; }
__device__ __forceinline__ int tap_dx(int tap) { return tap % 3 - 1; }

__device__ __forceinline__ void mma_bf16(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ size_t node_index(const uint32_t* base, int b, int H, int W, int i, int j) {
    const size_t b0 = base ? (size_t)base[b] : (size_t)b * (size_t)H * (size_t)W;
    return b0 + (size_t)i * W + j;
}

// ---------------------------------------------------------------------------
// weights: float masters -> bfloat16 layer copies (wk: [tap][out][in]; wt:
// the input-gradient form, wt[tap'][in][out] = W[8 - tap'][out][in]) and
// bfloat16-rounded floats for the first and last layers
__global__ void k_prep_weights(const float* __restrict__ master, bf16* wk, bf16* wt, float* w1r, float* w6r) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < 4 * 9 * CH * CH) {
        const int l = q / (9 * CH * CH), r = q % (9 * CH * CH);
        const int tap = r / (CH * CH), co = (r / CH) % CH, ci = r % CH;
        const bf16 v = __float2bfloat16_rn(master[off_w(l + 1) + r]);
        wk[q] = v;
        wt[l * 9 * CH * CH + ((8 - tap) * CH + ci) * CH + co] = v;
    }
    if (q < 9 * CH) {
        w1r[q] = __bfloat162float(__float2bfloat16_rn(master[off_w(0) + q]));
        w6r[q] = __bfloat162float(__float2bfloat16_rn(master[off_w(5) + q]));
    }
}

// ---------------------------------------------------------------------------
// a block's next tile of TY x CX nodes: sample and first node
struct Tile {
    int b, i0, j0;
};
__device__ __forceinline__ Tile tile_at(long long q, int tj, int ti) {
    const int b = (int)(q / ((long long)tj * ti)), r = (int)(q - (long long)b * tj * ti);
    return Tile{b, (r / tj) * TY, (r % tj) * CX};
}

// a tile of float nodes with its halo (zero outside the grid) in shared memory
__device__ __forceinline__ void stage_nodes(float* xs, const float* __restrict__ x, const uint32_t* base, const Tile& t,
                                            int H, int W) {
    for (int q = threadIdx.x; q < (TY + 2) * (CX + 2); q += blockDim.x) {
        const int hi = q / (CX + 2), hj = q - hi * (CX + 2);
        const int gi = t.i0 + hi - 1, gj = t.j0 + hj - 1;
        xs[q] = (gi >= 0 && gi < H && gj >= 0 && gj < W) ? x[node_index(base, t.b, H, W, gi, gj)] : 0.0f;
    }
}

// layer 1 (1 -> 32): a warp a tile row, a lane an output channel with its nine
// weights in registers, the row's 3 x 3 windows passing by in shared memory (three
// broadcast reads and nine operations a node and lane; a node's 64 bytes are one
// store of the warp).  513^2 nodes: 21 -> 10.5 us (a thread a node read 288 weights
// from shared memory and stored 64 bytes a lane).
__global__ void __launch_bounds__(32 * TY) k_conv1(const float* __restrict__ x, bf16* __restrict__ h,
                                                   const float* __restrict__ w1, const float* __restrict__ b1,
                                                   const uint32_t* __restrict__ base, int B, int H, int W) {
    __shared__ float xs[(TY + 2) * (CX + 2)];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    float w[9];
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) w[tap] = w1[tap * CH + lane];
    const float bias = b1[lane];
    const int tj = (W + CX - 1) / CX, ti = (H + TY - 1) / TY;
    const long long ntiles = (long long)B * tj * ti;
    for (long long q = blockIdx.x; q < ntiles; q += gridDim.x) {
        const Tile t = tile_at(q, tj, ti);
        __syncthreads();
        stage_nodes(xs, x, base, t, H, W);
        __syncthreads();
        const int i = t.i0 + row, nj = min(CX, W - t.j0);
        if (i >= H) continue;
        bf16* dst = h + node_index(base, t.b, H, W, i, t.j0) * CH + lane;
        const float* xr = xs + row * (CX + 2);
        float v[3][3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            v[d][1] = xr[d * (CX + 2)];
            v[d][2] = xr[d * (CX + 2) + 1];
        }
#pragma unroll 4
        for (int j = 0; j < nj; ++j) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                v[d][0] = v[d][1];
                v[d][1] = v[d][2];
                v[d][2] = xr[d * (CX + 2) + j + 2];
            }
            float a = bias;
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) a += w[tap] * v[tap / 3][tap % 3];
            dst[(size_t)j * CH] = __float2bfloat16_rn(fmaxf(a, 0.0f));
        }
    }
}

// ---------------------------------------------------------------------------
// four 8 x 8 matrices of bfloat16 from shared memory, a row address a lane
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const bf16* p) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}

// 16 bytes from global to shared memory without a register, zeros unless `in`
__device__ __forceinline__ void copy16(void* dst, const void* src, bool in) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// all but the latest N groups of copies have landed (this thread's)
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// a tile of rows x cols 32-channel nodes from node (i0, j0) on (zero outside the
// grid) into shared memory, asynchronously
__device__ __forceinline__ void stage_channels(bf16* xs, const bf16* __restrict__ in, size_t node0, int i0, int j0,
                                               int rows, int cols, int H, int W) {
    for (int q = threadIdx.x; q < rows * cols * 4; q += blockDim.x) {
        const int nd = q >> 2, part = q & 3;
        const int hi = nd / cols, hj = nd - hi * cols;
        const int gi = i0 + hi, gj = j0 + hj;
        const bool ok = gi >= 0 && gi < H && gj >= 0 && gj < W;
        copy16(&xs[nd * HP + part * 8], in + (ok ? (node0 + (size_t)gi * W + gj) * CH + part * 8 : 0), ok);
    }
    copy_commit();
}
__device__ __forceinline__ void stage_halo(bf16* xs, const bf16* __restrict__ in, const uint32_t* base, const Tile& t,
                                           int H, int W) {
    stage_channels(xs, in, node_index(base, t.b, H, W, 0, 0), t.i0 - 1, t.j0 - 1, TY + 2, CX + 2, H, W);
}
constexpr int TILE_ELEMS = (TY + 2) * (CX + 2) * HP;
constexpr int CONV_SMEM = 2 * TILE_ELEMS * 2;      // two tiles

// 32 -> 32 convolution on the tensor cores.  MODE 0: out = relu(conv + bias);
// MODE 1: out = conv where mask > 0, else 0 (input gradient through a ReLU).
// A warp takes 16 columns of the tile and 16 output channels, their weights in
// registers throughout (72), and marches down the staged rows: an ldmatrix of an
// input row's 16 nodes feeds six mma, the row above's, its own and the row
// below's by two channel octets, so that three rows of accumulators are open and a
// row is written when its last input row has passed.  The block's next tile is on
// its way while one is computed.  Shared-memory reads (twelve for four mma) and
// the latency of staging bounded the form before: 513^2 nodes 27 -> 20.5 us a layer
// (device time under ncu; the mma pipe 48 % busy).  Each output accumulates
// in the same order (taps, then channel halves).
template <int MODE>
__global__ void __launch_bounds__(CONV_THREADS, 4) k_conv32(const bf16* __restrict__ in, bf16* __restrict__ out,
                                                         const bf16* __restrict__ w, const float* __restrict__ bias,
                                                         const bf16* __restrict__ mask,
                                                         const uint32_t* __restrict__ base, int B, int H, int W) {
    extern __shared__ __align__(16) bf16 smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int cg = (warp >> 1) * 16, c0 = (warp & 1) * 16;     // first column and output channel
    uint32_t wb[9][2][2][2];
#pragma unroll
    for (int tap = 0; tap < 9; ++tap)
#pragma unroll
        for (int kh = 0; kh < 2; ++kh)
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                const uint32_t* p =
                    (const uint32_t*)(w + (size_t)(tap * CH + c0 + nt * 8 + g) * CH + kh * 16 + 2 * t);
                wb[tap][kh][nt][0] = __ldg(p);
                wb[tap][kh][nt][1] = __ldg(p + 4);
            }
    if (!chained()) return;                                   // (the weights are older than the kernel before)
    float bv[2][2] = {};
    if (MODE == 0)
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            bv[nt][0] = bias[c0 + nt * 8 + 2 * t];
            bv[nt][1] = bias[c0 + nt * 8 + 2 * t + 1];
        }
    // row addresses of the lane's matrices: nodes 0-7, 8-15 by channels 0-7, then 8-15
    const int xo = (cg + (lane & 15)) * HP + (lane >> 4) * 8;
    const int tj = (W + CX - 1) / CX, ti = (H + TY - 1) / TY;
    const long long ntiles = (long long)B * tj * ti;
    long long q = blockIdx.x;
    if (q < ntiles) stage_halo(smem, in, base, tile_at(q, tj, ti), H, W);
    for (int buf = 0; q < ntiles; q += gridDim.x, buf ^= 1) {
        const Tile tl = tile_at(q, tj, ti);
        if (q + gridDim.x < ntiles) {
            stage_halo(smem + (buf ^ 1) * TILE_ELEMS, in, base, tile_at(q + gridDim.x, tj, ti), H, W);
            copy_wait<1>();
        } else {
            copy_wait<0>();
        }
        __syncthreads();
        const bf16* xl = smem + buf * TILE_ELEMS + xo;
        const bool on = tl.j0 + cg < W;                   // (the warp's columns)
        float acc[3][2][4];
        // MODE 1: the mask of the next row to write, loaded a row ahead
        __nv_bfloat162 mk[2][2], mn[2][2];
        auto load_mask = [&](int r) {
#pragma unroll
            for (int half = 0; half < 2; ++half)
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    const int oi = tl.i0 + r, oj = tl.j0 + cg + g + 8 * half;
                    mn[half][nt] = __floats2bfloat162_rn(0.0f, 0.0f);
                    if (oi < H && oj < W)
                        mn[half][nt] = *(const __nv_bfloat162*)(mask + node_index(base, tl.b, H, W, oi, oj) * CH + c0 +
                                                                nt * 8 + 2 * t);
                }
        };
        if (MODE == 1) load_mask(0);
        if (on) {
#pragma unroll
        for (int hi = 0; hi < TY + 2; ++hi) {              // staged input row
            if (hi < TY)
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[hi % 3][nt][e] = 0.0f;
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                for (int kh = 0; kh < 2; ++kh) {
                    uint32_t a[4];
                    ldsm4(a, xl + (hi * (CX + 2) + dx) * HP + kh * 16);
#pragma unroll
                    for (int d = 0; d < 3; ++d) {          // tap row: output row hi - d
                        if (hi - d < 0 || hi - d >= TY) continue;
#pragma unroll
                        for (int nt = 0; nt < 2; ++nt)
                            mma_bf16(acc[(hi - d + 3) % 3][nt], a[0], a[1], a[2], a[3], wb[3 * d + dx][kh][nt][0],
                                     wb[3 * d + dx][kh][nt][1]);
                    }
                }
            if (hi < 2) continue;
            const int r = hi - 2, oi = tl.i0 + r;
            if (MODE == 1) {
#pragma unroll
                for (int half = 0; half < 2; ++half)
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt) mk[half][nt] = mn[half][nt];
                if (r + 1 < TY) load_mask(r + 1);
            }
            if (oi >= H) continue;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int oj = tl.j0 + cg + g + 8 * half;
                if (oj >= W) continue;
                const size_t nd = node_index(base, tl.b, H, W, oi, oj);
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    const int c = c0 + nt * 8 + 2 * t;
                    float v0 = acc[r % 3][nt][2 * half], v1 = acc[r % 3][nt][2 * half + 1];
                    if (MODE == 0) {
                        v0 = fmaxf(v0 + bv[nt][0], 0.0f);
                        v1 = fmaxf(v1 + bv[nt][1], 0.0f);
                    } else {
                        const __nv_bfloat162 m = mk[half][nt];
                        if (!(__bfloat162float(m.x) > 0.0f)) v0 = 0.0f;
                        if (!(__bfloat162float(m.y) > 0.0f)) v1 = 0.0f;
                    }
                    *(__nv_bfloat162*)(out + nd * CH + c) = __floats2bfloat162_rn(v0, v1);
                }
            }
        }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// layer 6 (32 -> 1) on the tensor cores: a warp 16 columns by four rows.  The
// three tap rows are three columns of one product, so that an input row's 16
// nodes (six ldmatrix, six mma) give what it adds to the output rows above, beside
// and below it; these meet by a shuffle and two additions.  The weights are
// bfloat16 values already, so the products are exact.  Each mma adds its 16 from
// zero and float additions join them: an mma does not round its addition to a
// running sum to nearest, and with the sum kept in it the layer's error against 64
// bits was 0.75 to 1.35 times that of a sum term by term, where it is now 0.45 to
// 0.95 (513^2 nodes, all layers: 96.4 -> 98.3 us).
// 513^2 nodes, all layers, before the launches overlapped: 115 us with a thread two
// nodes' 288 products on the CUDA cores, 107 us.
__global__ void __launch_bounds__(16 * TY) k_conv6(const bf16* __restrict__ h, float* __restrict__ y,
                                                   const float* __restrict__ w6, const float* __restrict__ b6,
                                                   const uint32_t* __restrict__ base, int B, int H, int W) {
    if (!chained()) return;
    static_assert(TY == 8 && CX == 32, "four warps: two column groups by two halves of the rows");
    __shared__ __align__(16) bf16 xs[TILE_ELEMS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int cg = (warp & 1) * 16, r0 = (warp >> 1) * (TY / 2);
    uint32_t wb[3][2][2];                                     // [dx][channel half]: column g is tap row g
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
        for (int kh = 0; kh < 2; ++kh)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float2 v = make_float2(0.0f, 0.0f);
                if (g < 3) v = *(const float2*)(w6 + (3 * g + dx) * CH + kh * 16 + 8 * e + 2 * t);
                const __nv_bfloat162 b = __floats2bfloat162_rn(v.x, v.y);
                wb[dx][kh][e] = *(const uint32_t*)&b;
            }
    const float bias = b6[0];
    const bf16* xl = xs + (r0 * (CX + 2) + cg + (lane & 15)) * HP + (lane >> 4) * 8;
    const int tj = (W + CX - 1) / CX, ti = (H + TY - 1) / TY;
    const long long ntiles = (long long)B * tj * ti;
    for (long long q = blockIdx.x; q < ntiles; q += gridDim.x) {
        const Tile tl = tile_at(q, tj, ti);
        __syncthreads();
        stage_halo(xs, h, base, tl, H, W);
        copy_wait<0>();
        __syncthreads();
        if (tl.j0 + cg >= W) continue;
        float o[3][2];                                        // open output rows: nodes g and g + 8 (lanes t = 0)
#pragma unroll
        for (int hi = 0; hi < TY / 2 + 2; ++hi) {
            float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                for (int kh = 0; kh < 2; ++kh) {
                    uint32_t a[4];
                    float p[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                    ldsm4(a, xl + (hi * (CX + 2) + dx) * HP + kh * 16);
                    mma_bf16(p, a[0], a[1], a[2], a[3], wb[dx][kh][0], wb[dx][kh][1]);
#pragma unroll
                    for (int e = 0; e < 4; ++e) c[e] += p[e];
                }
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const float below = __shfl_down_sync(0xFFFFFFFFu, c[2 * half], 1);      // tap row 2, of lane t = 1
                if (hi >= 2) o[(hi - 2) % 3][half] += below;
                if (hi >= 1 && hi - 1 < TY / 2) o[(hi - 1) % 3][half] += c[2 * half + 1];
                if (hi < TY / 2) o[hi % 3][half] = c[2 * half];
            }
            if (hi < 2) continue;
            const int i = tl.i0 + r0 + hi - 2;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int j = tl.j0 + cg + g + 8 * half;
                if (t == 0 && i < H && j < W) y[node_index(base, tl.b, H, W, i, j)] = o[(hi - 2) % 3][half] + bias;
            }
        }
    }
}

// The same in training, a thread two nodes (rows r and r + 4), summed tap by tap:
// the residual loss differentiates y twice, and its gradient (through bfloat16)
// shows the last bit of y at 2e-5.  So the y of a loss and the y of inference differ
// in the last bits.
__global__ void __launch_bounds__(16 * TY) k_conv6_train(const bf16* __restrict__ h, float* __restrict__ y,
                                                         const float* __restrict__ w6, const float* __restrict__ b6,
                                                         const uint32_t* __restrict__ base, int B, int H, int W) {
    __shared__ __align__(16) bf16 xs[(TY + 2) * (CX + 2) * HP];
    __shared__ __align__(16) float ws[9 * CH];
    for (int q = threadIdx.x; q < 9 * CH; q += blockDim.x) ws[q] = w6[q];
    const float bias = b6[0];
    const int row = threadIdx.x / CX, col = threadIdx.x % CX;
    const int tj = (W + CX - 1) / CX, ti = (H + TY - 1) / TY;
    const long long ntiles = (long long)B * tj * ti;
    for (long long q = blockIdx.x; q < ntiles; q += gridDim.x) {
        const Tile t = tile_at(q, tj, ti);
        __syncthreads();
        stage_halo(xs, h, base, t, H, W);
        copy_wait<0>();
        __syncthreads();
        const int j = t.j0 + col;
        float acc[2] = {bias, bias};
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
            const int i0 = t.i0 + row + tap_dy(tap), jj = j + tap_dx(tap);
            if (jj < 0 || jj >= W) continue;
            const uint4* src = (const uint4*)(xs + ((row + tap / 3) * (CX + 2) + col + tap % 3) * HP);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const float4 wa = *(const float4*)&ws[tap * CH + p * 8], wc = *(const float4*)&ws[tap * CH + p * 8 + 4];
                const float wv[8] = {wa.x, wa.y, wa.z, wa.w, wc.x, wc.y, wc.z, wc.w};
#pragma unroll
                for (int n = 0; n < 2; ++n) {
                    if (i0 + n * (TY / 2) < 0 || i0 + n * (TY / 2) >= H) continue;
                    const uint4 v = src[(size_t)n * (TY / 2) * (CX + 2) * HP / 8 + p];
                    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        acc[n] += wv[2 * e] * __uint_as_float(u[e] << 16);
                        acc[n] += wv[2 * e + 1] * __uint_as_float(u[e] & 0xFFFF0000u);
                    }
                }
            }
        }
        if (j >= W) continue;
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const int i = t.i0 + row + n * (TY / 2);
            if (i < H) y[node_index(base, t.b, H, W, i, j)] = acc[n];
        }
    }
}

// ---------------------------------------------------------------------------
// loss: g6 = 2 (y - t) / N and per-block partial sums of (y - t)^2
__global__ void __launch_bounds__(256) k_loss(const float* __restrict__ y, const float* __restrict__ t, float* g6,
                                              double* part, long long n) {
    double acc = 0.0;
    const float s = (float)(2.0 / (double)n);
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        const float d = y[p] - t[p];
        g6[p] = s * d;
        acc += (double)d * (double)d;
    }
    __shared__ double red[256];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// residual loss of a start on an r-z grid (dz = dr): the unit finite-volume
// coefficients of radial node j of W, and (S v)_ij on an interior row with
// rows 0 and H - 1 of v read as zero (Dirichlet)
__device__ __forceinline__ void rz_coeffs(int j, int W, float& ap, float& am, float& w) {
    const int nr = W - 1;
    ap = j < nr ? (float)j + 0.5f : 0.0f;
    am = j > 0 ? (float)j - 0.5f : 0.0f;
    w = j == 0 ? 0.125f : (j == nr ? 0.5f * (float)nr - 0.125f : (float)j);
}
__device__ __forceinline__ float rz_apply(const float* __restrict__ v, size_t k, int H, int W, int i, int j) {
    float ap, am, w;
    rz_coeffs(j, W, ap, am, w);
    float s = (ap + am + 2.0f * w) * v[k];
    if (j + 1 < W) s -= ap * v[k + 1];
    if (j > 0) s -= am * v[k - 1];
    if (i + 1 < H - 1) s -= w * v[k + W];
    if (i - 1 > 0) s -= w * v[k - W];
    return s;
}

// r = w x - S y on the interior rows (0 on the electrode rows) and
// per-block partial sums of r^2
__global__ void __launch_bounds__(256) k_rz_resid(const float* __restrict__ x, const float* __restrict__ y,
                                                  float* __restrict__ r, double* part, int B, int H, int W) {
    const long long n = (long long)B * H * W;
    double acc = 0.0;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        const int q = (int)(p % ((long long)H * W)), i = q / W, j = q - i * W;
        if (i == 0 || i == H - 1) {
            r[p] = 0.0f;
            continue;
        }
        float ap, am, w;
        rz_coeffs(j, W, ap, am, w);
        const float v = w * x[p] - rz_apply(y, (size_t)p, H, W, i, j);
        r[p] = v;
        acc += (double)v * (double)v;
    }
    __shared__ double red[256];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// g = scale S r on the interior rows, 0 on the electrode rows (S is
// symmetric, so this is scale S^T r)
__global__ void __launch_bounds__(256) k_rz_resid_grad(const float* __restrict__ r, float* __restrict__ g, float scale,
                                                       int B, int H, int W) {
    const long long n = (long long)B * H * W;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        const int q = (int)(p % ((long long)H * W)), i = q / W, j = q - i * W;
        g[p] = (i == 0 || i == H - 1) ? 0.0f : scale * rz_apply(r, (size_t)p, H, W, i, j);
    }
}

// the sum of a loss's n <= LOSS_BLOCKS partials in their order, by one block (a
// chain of double additions, 8 us: it runs beside k_wgrad_edge's blocks)
__device__ __forceinline__ void loss_sum(const double* __restrict__ part, int n, double inv_count, double* out,
                                         double* p) {
    if ((int)threadIdx.x < n) p[threadIdx.x] = part[threadIdx.x];
    __syncthreads();
    if (threadIdx.x != 0) return;
    double s = 0.0;
#pragma unroll 8
    for (int q = 0; q < n; ++q) s += p[q];
    *out = s * inv_count;
}

// gradient with respect to a_5: (sum_tap w6[tap][c] g6[p - tap]) where h5 > 0, a
// lane a channel as in k_conv1 (129^2 nodes, eight samples: 13.8 -> 11.4 us)
__global__ void __launch_bounds__(32 * TY) k_conv6_bwd(const float* __restrict__ g6, const bf16* __restrict__ h5,
                                                       bf16* __restrict__ g5, const float* __restrict__ w6, int B,
                                                       int H, int W) {
    __shared__ float xs[(TY + 2) * (CX + 2)];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    float w[9];
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) w[tap] = w6[tap * CH + lane];
    const int tj = (W + CX - 1) / CX, ti = (H + TY - 1) / TY;
    const long long ntiles = (long long)B * tj * ti;
    for (long long q = blockIdx.x; q < ntiles; q += gridDim.x) {
        const Tile t = tile_at(q, tj, ti);
        __syncthreads();
        stage_nodes(xs, g6, nullptr, t, H, W);
        __syncthreads();
        const int i = t.i0 + row, nj = min(CX, W - t.j0);
        if (i >= H) continue;
        const size_t p0 = node_index(nullptr, t.b, H, W, i, t.j0) * CH + lane;
        const float* xr = xs + row * (CX + 2);
#pragma unroll 4
        for (int j = 0; j < nj; ++j) {
            const bf16 m = h5[p0 + (size_t)j * CH];
            float a = 0.0f;
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) a += w[tap] * xr[(2 - tap / 3) * (CX + 2) + j + 2 - tap % 3];
            if (!(__bfloat162float(m) > 0.0f)) a = 0.0f;
            g5[p0 + (size_t)j * CH] = __float2bfloat16_rn(a);
        }
    }
}

// ---------------------------------------------------------------------------
// Weight gradients of the first and last layers (CUDA cores): each tap's sum over
// the nodes of a node value at the tap's place (layer 1: x at p + tap, layer 6: g6
// at p - tap) times 32 channel values at p (g1, h5).  A warp takes a row of an 8 x
// 16 node tile, a lane a channel with its nine sums in registers, the node values
// staged in shared memory and read as broadcasts; the rows' sums meet at the end
// (a thread a tap and channel read two words of shared memory a product, which
// bounded it, 21 us each at eight samples of 129^2 nodes: a step 380 -> 364 us).  Partials: 288
// weights, then the bias gradients.  Layer 6: a last block sums the loss.
template <int LAYER>
__global__ void __launch_bounds__(32 * TY) k_wgrad_edge(const float* __restrict__ nodes, const bf16* __restrict__ chan,
                                                        float* part, int B, int H, int W,
                                                        const double* __restrict__ lpart, int lb, double inv_count,
                                                        double* lsum) {
    __shared__ float xs[(TY + 2) * (TX + 2)];
    __shared__ __align__(16) float red[10][TY][CH];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5, nblk = (int)gridDim.x - (LAYER == 6 ? 1 : 0);
    if (LAYER == 6 && (int)blockIdx.x == nblk) {
        static_assert(LOSS_BLOCKS <= 32 * TY && sizeof(red) >= LOSS_BLOCKS * sizeof(double), "loss_sum");
        loss_sum(lpart, lb, inv_count, lsum, reinterpret_cast<double*>(&red[0][0][0]));
        return;
    }
    const int tj = (W + TX - 1) / TX, ti = (H + TY - 1) / TY;
    const long long ntiles = (long long)B * tj * ti, n = (long long)H * W;
    float acc[10] = {};                                       // the taps, the bias
    for (long long tile = blockIdx.x; tile < ntiles; tile += nblk) {
        const int b = (int)(tile / ((long long)tj * ti));
        const int r = (int)(tile - (long long)b * tj * ti);
        const int i0 = (r / tj) * TY, j0 = (r % tj) * TX, i = i0 + row, nj = min(TX, W - j0);
        float v[TX];
        if (i < H) {
            const bf16* src = chan + ((size_t)b * n + (size_t)i * W + j0) * CH + lane;
#pragma unroll
            for (int j = 0; j < TX; ++j) v[j] = j < nj ? __bfloat162float(src[(size_t)j * CH]) : 0.0f;
        }
        __syncthreads();
        for (int q = threadIdx.x; q < (TY + 2) * (TX + 2); q += blockDim.x) {
            const int gi = i0 + q / (TX + 2) - 1, gj = j0 + q % (TX + 2) - 1;
            xs[q] = (gi >= 0 && gi < H && gj >= 0 && gj < W) ? nodes[(size_t)b * n + (size_t)gi * W + gj] : 0.0f;
        }
        __syncthreads();
        if (i >= H) continue;
        const float* xr = xs + row * (TX + 2);
#pragma unroll
        for (int j = 0; j < TX; ++j) {
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
                const int y = LAYER == 1 ? tap / 3 : 2 - tap / 3, x = LAYER == 1 ? tap % 3 : 2 - tap % 3;
                acc[tap] += v[j] * xr[y * (TX + 2) + j + x];
            }
            if (LAYER == 1) acc[9] += v[j];
        }
        if (LAYER == 6 && lane < TX) acc[9] += xr[TX + 2 + lane + 1];
    }
#pragma unroll
    for (int k = 0; k < 10; ++k) red[k][row][lane] = acc[k];
    __syncthreads();
    float* out = part + (size_t)blockIdx.x * PART_STRIDE;
    for (int q = threadIdx.x; q < (LAYER == 1 ? 10 : 9) * CH; q += blockDim.x) {
        float t = 0.0f;
#pragma unroll
        for (int w = 0; w < TY; ++w) t += red[q / CH][w][q % CH];
        out[q] = t;
    }
    if (LAYER == 6 && row == 0) {
        float t = 0.0f;
#pragma unroll
        for (int w = 0; w < TY; ++w) t += red[9][w][lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
        if (lane == 0) out[9 * CH] = t;
    }
}

// the same, each 8 x 8 matrix transposed
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const bf16* p) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}

// weight gradient of a 32 -> 32 layer on the tensor cores: warp = tap.  Both
// operands have the nodes as the GEMM's k: the tiles are staged as they lie
// (node-major) and read through transposing ldmatrix, four for eight mma, where a
// tap's shift is an offset of nodes.  (Staged channel-major by 2-byte stores with
// bank conflicts and read by 2-byte loads: 129^2 nodes, eight samples, 27 -> 18.5 us.)
__global__ void __launch_bounds__(288) k_wgrad32(const bf16* __restrict__ h, const bf16* __restrict__ g,
                                                 float* part, int B, int H, int W) {
    __shared__ __align__(16) bf16 gs[TY * TX * HP];
    __shared__ __align__(16) bf16 hs[(TY + 2) * (TX + 2) * HP];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gq = lane >> 2, t = lane & 3;
    const int dy = tap_dy(warp), dx = tap_dx(warp);
    // row addresses of the lane's matrices.  A (output channels by nodes): nodes
    // 0-7 by channels 0-7, 8-15, then nodes 8-15; B (nodes by input channels):
    // channels 0-7 by nodes 0-7, 8-15, then channels 8-15
    const bf16* ga = gs + ((lane & 7) + (lane >> 4) * 8) * HP + ((lane >> 3) & 1) * 8;
    const bf16* hb = hs + ((dy + 1) * (TX + 2) + dx + 1 + (lane & 7) + ((lane >> 3) & 1) * 8) * HP + (lane >> 4) * 8;
    float acc[2][4][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[mt][nt][e] = 0.0f;
    float bacc = 0.0f;
    const int tj = (W + TX - 1) / TX, ti = (H + TY - 1) / TY;
    const long long ntiles = (long long)B * tj * ti;
    const long long n = (long long)H * W;
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int b = (int)(tile / ((long long)tj * ti));
        const int r = (int)(tile - (long long)b * tj * ti);
        const int i0 = (r / tj) * TY, j0 = (r % tj) * TX;
        __syncthreads();
        stage_channels(gs, g, (size_t)b * n, i0, j0, TY, TX, H, W);
        stage_channels(hs, h, (size_t)b * n, i0 - 1, j0 - 1, TY + 2, TX + 2, H, W);
        copy_wait<0>();
        __syncthreads();
#pragma unroll
        for (int ri = 0; ri < TY; ++ri) {
            uint32_t a[2][4], bb[2][4];
            ldsm4t(a[0], ga + ri * TX * HP);
            ldsm4t(a[1], ga + ri * TX * HP + 16);
            ldsm4t(bb[0], hb + ri * (TX + 2) * HP);
            ldsm4t(bb[1], hb + ri * (TX + 2) * HP + 16);
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
                    mma_bf16(acc[mt][nt], a[mt][0], a[mt][1], a[mt][2], a[mt][3], bb[nt >> 1][2 * (nt & 1)],
                             bb[nt >> 1][2 * (nt & 1) + 1]);
        }
        if (threadIdx.x < CH)
#pragma unroll 32
            for (int nd = 0; nd < TY * TX; ++nd) bacc += __bfloat162float(gs[nd * HP + threadIdx.x]);
    }
    float* P = part + (size_t)blockIdx.x * PART_STRIDE;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const int co = mt * 16 + gq, ci = nt * 8 + 2 * t;
            P[(warp * CH + co) * CH + ci] = acc[mt][nt][0];
            P[(warp * CH + co) * CH + ci + 1] = acc[mt][nt][1];
            P[(warp * CH + co + 8) * CH + ci] = acc[mt][nt][2];
            P[(warp * CH + co + 8) * CH + ci + 1] = acc[mt][nt][3];
        }
    if (threadIdx.x < CH) P[9 * CH * CH + threadIdx.x] = bacc;
}

// out[k] = sum over blocks c (in order) of part[c * PART_STRIDE + k], k < NP: a block
// brings 32 values' partials into shared memory with all its loads in flight, a
// warp adds them in order (the chain of additions waited for a load each: 304
// partials of 9248 values 31 -> 10 us).  One launch for all layers: a layer's fills
// a quarter of the SMs for 10 us, six of them 60 us of a step: 8 x 129^2 nodes 411
// -> 380 us a step (and, with no more blocks than tiles, 1 x 33 x 47 nodes 245 -> 192 us).
constexpr int RED_COLS = 32;
__global__ void __launch_bounds__(256) k_reduce(const float* __restrict__ part, int nblocks, float* out) {
    extern __shared__ float ps[];
    const int k0 = blockIdx.x * RED_COLS, lane = threadIdx.x & 31;
    const bool in = k0 + lane < NP;
#pragma unroll 8
    for (int c = threadIdx.x >> 5; c < nblocks; c += 8)
        ps[c * RED_COLS + lane] = in ? part[(size_t)c * PART_STRIDE + k0 + lane] : 0.0f;
    __syncthreads();
    if (threadIdx.x >= RED_COLS || !in) return;
    float s = 0.0f;
#pragma unroll 16
    for (int c = 0; c < nblocks; ++c) s += ps[c * RED_COLS + lane];
    out[k0 + lane] = s;
}

__global__ void k_adam(float* w, float* m, float* v, const float* __restrict__ g, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= NP) return;
    const float gq = g[q];
    const float mq = b1 * m[q] + (1.0f - b1) * gq;
    const float vq = b2 * v[q] + (1.0f - b2) * gq * gq;
    m[q] = mq;
    v[q] = vq;
    w[q] -= lr * (mq / c1) / (sqrtf(vq / c2) + eps);
}

}  // namespace
}  // namespace pd

using namespace pd;

struct pd_net {
    int64_t max_nodes;
    cudaStream_t stream;
    int sms;
    float *master, *m, *v, *grad;
    bf16 *wk, *wt;
    float *w1r, *w6r;
    bf16* h[5];
    bf16* g[5];
    float *g6, *ybuf;
    float* part;
    double *lpart, *lsum;
    int64_t adam_k;
    bool have_grad;
    std::string err;
};

namespace {

struct NetLayout {
    size_t master, m, v, grad, wk, wt, w1r, w6r, h[5], g[5], g6, ybuf, part, lpart, lsum, total;
};

NetLayout net_layout(int64_t max_nodes) {
    NetLayout L;
    size_t o = 0;
    auto take = [&](size_t b) {
        const size_t r = o;
        o += al(b);
        return r;
    };
    L.master = take(NP * 4);
    L.m = take(NP * 4);
    L.v = take(NP * 4);
    L.grad = take(NP * 4);
    L.wk = take(4 * 9 * CH * CH * 2);
    L.wt = take(4 * 9 * CH * CH * 2);
    L.w1r = take(9 * CH * 4);
    L.w6r = take(9 * CH * 4);
    for (int l = 0; l < 5; ++l) L.h[l] = take((size_t)max_nodes * CH * 2);
    for (int l = 0; l < 5; ++l) L.g[l] = take((size_t)max_nodes * CH * 2);
    L.g6 = take((size_t)max_nodes * 4);
    L.ybuf = take((size_t)max_nodes * 4);
    L.part = take((size_t)MAX_PART_BLOCKS * PART_STRIDE * 4);
    L.lpart = take(LOSS_BLOCKS * 8);
    L.lsum = take(8);
    L.total = o;
    return L;
}

// blocks of the weight gradients over their tiles of TY x TX nodes
int part_blocks(const pd_net* net, int B, int H, int W) {
    const long long n = (long long)B * ((W + TX - 1) / TX) * ((H + TY - 1) / TY);
    return (int)std::min<long long>(n, std::min(MAX_PART_BLOCKS, 2 * net->sms));
}
int elem_blocks(const pd_net* net, long long n) {
    const long long b = (n + 255) / 256;
    return (int)std::max(1LL, std::min(b, (long long)net->sms * 16));
}

pd_status net_fail(pd_net* net, pd_status code, const std::string& msg) {
    if (net) net->err = msg;
    return code;
}

bool shape_ok(const pd_net* net, int B, int H, int W) {
    return B >= 1 && H >= 1 && W >= 1 && (int64_t)B * H * W <= net->max_nodes;
}

// blocks of a kernel over the tiles of TY x CX nodes, `per_sm` to an SM
int tile_blocks(const pd_net* net, int B, int H, int W, int per_sm) {
    const long long n = (long long)B * ((W + CX - 1) / CX) * ((H + TY - 1) / TY);
    return (int)std::min(n, (long long)net->sms * per_sm);
}

// each layer's blocks start, and read its weights, while the layer before ends:
// 513^2 nodes 107 -> 96 us.  Not in training: a step of 8 x 129^2 nodes 408 us,
// 412 with these layers launched so, 435 with the back-propagation too.
void forward_layers(pd_net* net, const float* x, float* y, int B, int H, int W, const uint32_t* base,
                    cudaStream_t s, bool training) {
    const float* P = net->master;
    const int gc = tile_blocks(net, B, H, W, 4), ge = tile_blocks(net, B, H, W, 8);
    k_conv1<<<ge, 32 * TY, 0, s>>>(x, net->h[0], net->w1r, P + off_b(0), base, B, H, W);
    for (int l = 1; l <= 4; ++l)
        launch(!training, k_conv32<0>, gc, CONV_THREADS, CONV_SMEM, s, net->h[l - 1], net->h[l],
               net->wk + (size_t)(l - 1) * 9 * CH * CH, P + off_b(l), nullptr, base, B, H, W);
    if (training) k_conv6_train<<<ge, 16 * TY, 0, s>>>(net->h[4], y, net->w6r, P + off_b(5), base, B, H, W);
    else launch(true, k_conv6, ge, 16 * TY, 0, s, net->h[4], y, net->w6r, P + off_b(5), base, B, H, W);
}

pd_status upload_weights(pd_net* net) {
    k_prep_weights<<<(4 * 9 * CH * CH + 255) / 256, 256, 0, net->stream>>>(net->master, net->wk, net->wt, net->w1r,
                                                                          net->w6r);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PD_OK : net_fail(net, PD_ERR_CUDA, cudaGetErrorString(e));
}

}  // namespace

namespace pd {
int net_forward_at(pd_net* net, const float* x, float* y, int B, int H, int W, const uint32_t* base,
                   int64_t node_span, cudaStream_t stream) {
    if (!net || node_span > net->max_nodes) return 1;
    forward_layers(net, x, y, B, H, W, base, stream, false);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}
int64_t net_max_nodes(const pd_net* net) { return net ? net->max_nodes : 0; }
}  // namespace pd

extern "C" {

pd_status pd_net_workspace_size(int64_t max_nodes, size_t* bytes) {
    if (!bytes || max_nodes < 1 || max_nodes > (int64_t)1 << 31) return PD_ERR_ARG;
    *bytes = net_layout(max_nodes).total;
    return PD_OK;
}

pd_status pd_net_create(int64_t max_nodes, void* ws, size_t bytes, void* stream, pd_net** out) {
    if (!out) return PD_ERR_ARG;
    *out = nullptr;
    if (max_nodes < 1 || max_nodes > (int64_t)1 << 31 || !ws || ((uintptr_t)ws & 255)) return PD_ERR_ARG;
    const NetLayout L = net_layout(max_nodes);
    if (bytes < L.total) return PD_ERR_ARG;
    pd_net* net = new (std::nothrow) pd_net();
    if (!net) return PD_ERR_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&net->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(k_conv32<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, CONV_SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(k_conv32<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, CONV_SMEM) != cudaSuccess) {
        delete net;
        return PD_ERR_CUDA;
    }
    char* w = (char*)ws;
    net->max_nodes = max_nodes;
    net->stream = (cudaStream_t)stream;
    net->master = (float*)(w + L.master);
    net->m = (float*)(w + L.m);
    net->v = (float*)(w + L.v);
    net->grad = (float*)(w + L.grad);
    net->wk = (bf16*)(w + L.wk);
    net->wt = (bf16*)(w + L.wt);
    net->w1r = (float*)(w + L.w1r);
    net->w6r = (float*)(w + L.w6r);
    for (int l = 0; l < 5; ++l) {
        net->h[l] = (bf16*)(w + L.h[l]);
        net->g[l] = (bf16*)(w + L.g[l]);
    }
    net->g6 = (float*)(w + L.g6);
    net->ybuf = (float*)(w + L.ybuf);
    net->part = (float*)(w + L.part);
    net->lpart = (double*)(w + L.lpart);
    net->lsum = (double*)(w + L.lsum);
    net->adam_k = 0;
    net->have_grad = false;
    if (cudaMemsetAsync(w, 0, L.g6, net->stream) != cudaSuccess || upload_weights(net) != PD_OK ||
        cudaStreamSynchronize(net->stream) != cudaSuccess) {
        delete net;
        return PD_ERR_CUDA;
    }
    *out = net;
    return PD_OK;
}

void pd_net_destroy(pd_net* net) {
    if (!net) return;
    cudaStreamSynchronize(net->stream);
    delete net;
}

pd_status pd_net_set_params(pd_net* net, const float* params) {
    if (!net || !params) return PD_ERR_ARG;
    if (cudaMemcpyAsync(net->master, params, NP * 4, cudaMemcpyHostToDevice, net->stream) != cudaSuccess ||
        cudaMemsetAsync(net->m, 0, NP * 4, net->stream) != cudaSuccess ||
        cudaMemsetAsync(net->v, 0, NP * 4, net->stream) != cudaSuccess)
        return net_fail(net, PD_ERR_CUDA, "parameter upload failed");
    net->adam_k = 0;
    net->have_grad = false;
    const pd_status r = upload_weights(net);
    if (r != PD_OK) return r;
    return cudaStreamSynchronize(net->stream) == cudaSuccess ? PD_OK : net_fail(net, PD_ERR_CUDA, "sync failed");
}

pd_status pd_net_get_params(pd_net* net, float* params) {
    if (!net || !params) return PD_ERR_ARG;
    if (cudaMemcpyAsync(params, net->master, NP * 4, cudaMemcpyDeviceToHost, net->stream) != cudaSuccess ||
        cudaStreamSynchronize(net->stream) != cudaSuccess)
        return net_fail(net, PD_ERR_CUDA, "parameter download failed");
    return PD_OK;
}

pd_status pd_net_forward(pd_net* net, const float* x, int B, int H, int W, float* y) {
    if (!net || !x || !y) return PD_ERR_ARG;
    if (!shape_ok(net, B, H, W)) return net_fail(net, PD_ERR_ARG, "batch exceeds the network's node capacity");
    forward_layers(net, x, y, B, H, W, nullptr, net->stream, false);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PD_OK : net_fail(net, PD_ERR_CUDA, cudaGetErrorString(e));
}

}  // extern "C"

namespace {

// back-propagation of the output gradient g6 (B H W floats) to the
// parameter gradient, and the loss (of lb partials) and gradient out to the host
// if asked
pd_status backprop(pd_net* net, const float* x, const float* g6, int B, int H, int W, int lb, double inv_count,
                   double* loss, float* grads) {
    cudaStream_t s = net->stream;
    const int pb = part_blocks(net, B, H, W);
    const int gc = tile_blocks(net, B, H, W, 4), ge = tile_blocks(net, B, H, W, 8);
    // layer 6
    k_wgrad_edge<6><<<pb + 1, 32 * TY, 0, s>>>(g6, net->h[4], net->part + off_w(5), B, H, W, net->lpart, lb, inv_count,
                                               net->lsum);
    k_conv6_bwd<<<ge, 32 * TY, 0, s>>>(g6, net->h[4], net->g[4], net->w6r, B, H, W);
    // layers 5 .. 2
    for (int l = 4; l >= 1; --l) {
        // weights then biases: both contiguous in the parameter vector
        k_wgrad32<<<pb, 288, 0, s>>>(net->h[l - 1], net->g[l], net->part + off_w(l), B, H, W);
        k_conv32<1><<<gc, CONV_THREADS, CONV_SMEM, s>>>(net->g[l], net->g[l - 1], net->wt + (size_t)(l - 1) * 9 * CH * CH,
                                                   nullptr, net->h[l - 1], nullptr, B, H, W);
    }
    // layer 1
    k_wgrad_edge<1><<<pb, 32 * TY, 0, s>>>(x, net->g[0], net->part + off_w(0), B, H, W, nullptr, 0, 0.0, nullptr);
    k_reduce<<<(NP + RED_COLS - 1) / RED_COLS, 256, (size_t)pb * RED_COLS * 4, s>>>(net->part, pb, net->grad);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return net_fail(net, PD_ERR_CUDA, cudaGetErrorString(e));
    net->have_grad = true;
    if (loss) e = cudaMemcpyAsync(loss, net->lsum, 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && grads) e = cudaMemcpyAsync(grads, net->grad, NP * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && (loss || grads)) e = cudaStreamSynchronize(s);
    return e == cudaSuccess ? PD_OK : net_fail(net, PD_ERR_CUDA, cudaGetErrorString(e));
}

}  // namespace

extern "C" {

pd_status pd_net_loss_grad(pd_net* net, const float* x, const float* t, int B, int H, int W, double* loss,
                           float* grads) {
    if (!net || !x || !t) return PD_ERR_ARG;
    if (!shape_ok(net, B, H, W)) return net_fail(net, PD_ERR_ARG, "batch exceeds the network's node capacity");
    cudaStream_t s = net->stream;
    const long long total = (long long)B * H * W;
    forward_layers(net, x, net->ybuf, B, H, W, nullptr, s, true);
    const int lb = (int)std::min<long long>(LOSS_BLOCKS, (total + 255) / 256);
    k_loss<<<lb, 256, 0, s>>>(net->ybuf, t, net->g6, net->lpart, total);
    return backprop(net, x, net->g6, B, H, W, lb, 1.0 / (double)total, loss, grads);
}

pd_status pd_net_loss_grad_rz(pd_net* net, const float* x, int B, int H, int W, double* loss, float* grads) {
    if (!net || !x) return PD_ERR_ARG;
    if (!shape_ok(net, B, H, W) || H < 3 || W < 2)
        return net_fail(net, PD_ERR_ARG, "batch exceeds the network's node capacity, or a grid below 3 x 2 nodes");
    cudaStream_t s = net->stream;
    const long long total = (long long)B * H * W, n_int = (long long)B * (H - 2) * W;
    forward_layers(net, x, net->ybuf, B, H, W, nullptr, s, true);
    const int lb = (int)std::min<long long>(LOSS_BLOCKS, (total + 255) / 256);
    // r into g6, then dL/dy = -(2 / N) S r into ybuf (y is not needed after r)
    k_rz_resid<<<lb, 256, 0, s>>>(x, net->ybuf, net->g6, net->lpart, B, H, W);
    k_rz_resid_grad<<<elem_blocks(net, total), 256, 0, s>>>(net->g6, net->ybuf, (float)(-2.0 / (double)n_int), B, H,
                                                           W);
    return backprop(net, x, net->ybuf, B, H, W, lb, 1.0 / (double)n_int, loss, grads);
}

pd_status pd_net_adam(pd_net* net, float lr, float b1, float b2, float eps) {
    if (!net) return PD_ERR_ARG;
    if (!net->have_grad) return net_fail(net, PD_ERR_STATE, "no gradient: call pd_net_loss_grad first");
    if (!(lr > 0) || !(b1 >= 0 && b1 < 1) || !(b2 >= 0 && b2 < 1) || !(eps >= 0))
        return net_fail(net, PD_ERR_ARG, "bad Adam hyper-parameters");
    net->adam_k += 1;
    const float c1 = (float)(1.0 - std::pow((double)b1, (double)net->adam_k));
    const float c2 = (float)(1.0 - std::pow((double)b2, (double)net->adam_k));
    k_adam<<<(NP + 255) / 256, 256, 0, net->stream>>>(net->master, net->m, net->v, net->grad, lr, b1, b2, eps, c1,
                                                      c2);
    return upload_weights(net);
}

}  // extern "C"
