// Warm-start MLP 16 -> 64 -> 64 -> 64 -> n_out (n_out <= 3, ReLU), BF16 tensor-core GEMMs with
// FP32 accumulation (mma.sync m16n8k16), training by hand-written backward
// kernels and Adam.
//
// Parameters are kept in FP32 ("master") in the packed order W1[16][64], b1,
// W2[64][64], b2, W3[64][64], b3, W4[64][n_out], b4 (y = x W + b per layer).
// Whoever writes a parameter also writes its BF16 copy in the network's weight
// image ([out][in] rows, padded), so a block copies all its weights as they
// lie; the transposed operands of the backward pass come from the same
// rows through transposing fragment loads.  Rounding points: the features and
// every hidden activation (after bias and ReLU) are rounded to BF16 where they
// become an MMA operand; the output error and every hidden error likewise.
// Accumulation and biases are FP32.
//
// Forward: one warp per 16-row tile; a layer's FP32 accumulator fragments are
// re-packed in registers as the next layer's A fragments.
// Gradients: blocks of 8 warps take up to 128 rows a round: each warp runs 16
// rows forward and back through the layers (dX = dZ W^T), leaving activations
// and errors in shared memory as [row][feature] BF16 pairs; then every warp
// owns some output tiles of dW = H^T dZ and adds the round's rows to them in
// registers (64 rows to an MMA chain, the chains added in FP32; no atomics),
// while the bias columns are summed by the threads.  Each block writes its FP32
// partial gradient once; the second kernel adds the partials in a fixed order
// and, in training, takes the Adam step and refreshes the weight image, so the
// result is reproducible run to run.
//
// What bounds a training step of 65,536 rows (3.7 GFLOP): the layer chain of a
// 16-row tile is a few hundred dependent instructions, so the rate follows the
// warps an SM runs side by side and what they do besides MMAs.  Four warps an
// SM (143 KB of shared memory a block for two weight copies and gradient
// accumulators), 2-byte transposed staging stores, dW accumulated in shared
// memory, uncoalesced weight conversion in every block and 304 partials summed
// one after the other took 133 us a step; this form took 36 us, and 34 us since
// a round's rows are drawn and read while the round before adds its dW (twelve
// warps a block, 168 registers, took 37 us).
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "kernels.h"
#include "launch_util.cuh"
#include "mlbm_internal.h"
#include "ring.cuh"
#include "step_node.cuh"

namespace mlbm {
namespace mlp {

constexpr int kIn = 16, kH = 64, kMaxOut = 3;
// packed offsets
constexpr int oW1 = 0, oB1 = oW1 + kIn * kH, oW2 = oB1 + kH, oB2 = oW2 + kH * kH, oW3 = oB2 + kH,
              oB3 = oW3 + kH * kH, oW4 = oB3 + kH;
// offset of b4 and parameter count for `no` outputs (9538 for no = 2)
__host__ __device__ constexpr int off_b4(int no) { return oW4 + kH * no; }
__host__ __device__ constexpr int param_count(int no) { return off_b4(no) + no; }
static_assert(param_count(2) == 9538, "packing");

// padded row strides (BF16 elements) that keep fragment loads free of bank conflicts
constexpr int kS16 = 24, kS64 = 72;

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void mma(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// four 8x8 BF16 matrices (TRANS: transposed); lane i gives the address of row
// i % 8 of matrix i / 8
template <bool TRANS>
__device__ __forceinline__ void ldsm4(uint32_t* r, const __nv_bfloat16* p) {
    const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p));
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}

// Weight image: [out][in] BF16 rows with padded strides (outputs padded to 8),
// FP32 biases; padding is zero.
struct __align__(16) Image {
    __nv_bfloat16 wt1[kH * kS16];
    __nv_bfloat16 wt2[kH * kS64];
    __nv_bfloat16 wt3[kH * kS64];
    __nv_bfloat16 wt4[8 * kS64];
    float b1[kH], b2[kH], b3[kH], b4[8];
};
static_assert(sizeof(Image) % 16 == 0, "copied 16 bytes at a time");

// parameter i (packed order) into the image
__device__ __forceinline__ void image_put(Image* I, int no, int i, float v) {
    const __nv_bfloat16 w = __float2bfloat16_rn(v);
    if (i < oB1) I->wt1[(i % kH) * kS16 + i / kH] = w;
    else if (i < oW2) I->b1[i - oB1] = v;
    else if (i < oB2) I->wt2[((i - oW2) % kH) * kS64 + (i - oW2) / kH] = w;
    else if (i < oW3) I->b2[i - oB2] = v;
    else if (i < oB3) I->wt3[((i - oW3) % kH) * kS64 + (i - oW3) / kH] = w;
    else if (i < oW4) I->b3[i - oB3] = v;
    else if (i < off_b4(no)) I->wt4[((i - oW4) % no) * kS64 + (i - oW4) / no] = w;
    else I->b4[i - off_b4(no)] = v;
}

// the image of new parameters, and Adam's moments back at zero
__global__ void take_params(int kp, int no, const float* __restrict__ P, Image* __restrict__ I, float* __restrict__ m,
                            float* __restrict__ v) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kp) return;
    image_put(I, no, i, P[i]);
    m[i] = 0.f;
    v[i] = 0.f;
}

// The image into the block's shared memory, 16 bytes a thread at a time past the
// registers.  Unlike a bulk copy on a barrier it needs no wait that could run
// out.
__device__ __forceinline__ void fetch_image(Image* s, const Image* I) {
    const uint32_t to = dev::saddr(s);
    for (uint32_t o = threadIdx.x * 16; o < sizeof(Image); o += blockDim.x * 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + o),
                     "l"(reinterpret_cast<const uint8_t*>(I) + o) : "memory");
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

// Row of the data set that minibatch row r reads: r itself (seed 0), else a
// splitmix64 hash of (seed, step, r) reduced modulo n_data.
__device__ __forceinline__ int64_t data_row(int64_t r, int64_t n_data, uint64_t seed, uint64_t step) {
    if (seed == 0) return r;
    uint64_t z = seed ^ (step * 0xD1B54A32D192ED03ull) ^ ((uint64_t)r * 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (int64_t)(z % (uint64_t)n_data);
}

// this lane's features of the tile (rows g, g + 8 of the warp's 16 rows);
// src0 / src1: data rows of those two rows, -1 for padding
__device__ __forceinline__ void read_x(const float* __restrict__ X, int64_t src0, int64_t src1, int t, float* v) {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = 0.f;
    if (src0 >= 0) {
        const float* x = X + src0 * kIn;
        v[0] = x[2 * t]; v[1] = x[2 * t + 1];
        v[4] = x[2 * t + 8]; v[5] = x[2 * t + 9];
    }
    if (src1 >= 0) {
        const float* x = X + src1 * kIn;
        v[2] = x[2 * t]; v[3] = x[2 * t + 1];
        v[6] = x[2 * t + 8]; v[7] = x[2 * t + 9];
    }
}

// ... and as an A fragment
__device__ __forceinline__ void pack_x(const float* v, uint32_t* a) {
    a[0] = pack2(v[0], v[1]);
    a[1] = pack2(v[2], v[3]);
    a[2] = pack2(v[4], v[5]);
    a[3] = pack2(v[6], v[7]);
}

// one hidden layer: A (k-tiles of the input) -> ReLU(A W + b) packed as the
// next A fragments
template <int KT>
__device__ __forceinline__ void hidden_layer(const uint32_t (*a)[4], const __nv_bfloat16* wt, int stride,
                                             const float* bias, int lane, uint32_t (*out)[4]) {
    const int t = lane & 3;
    // row of an 8x8 matrix, and which half (KT = 1: which n-tile and half) of the k-tiles it belongs to
    const __nv_bfloat16* row = wt + (lane & 7) * stride;
    const int sel = lane >> 3;
#pragma unroll
    for (int np = 0; np < 4; ++np) {  // pairs of n-tiles
        float d[2][4];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float2 bb = *reinterpret_cast<const float2*>(bias + 16 * np + 8 * j + 2 * t);
            d[j][0] = bb.x; d[j][1] = bb.y; d[j][2] = bb.x; d[j][3] = bb.y;
        }
        if (KT == 1) {
            uint32_t b[4];  // n-tile 0 halves, n-tile 1 halves
            ldsm4<false>(b, row + (16 * np + 8 * (sel >> 1)) * stride + 8 * (sel & 1));
            mma(d[0], a[0], b[0], b[1]);
            mma(d[1], a[0], b[2], b[3]);
        } else {
#pragma unroll
            for (int kp = 0; kp < KT / 2; ++kp) {
                uint32_t b0[4], b1[4];  // k-tile 2 kp halves, k-tile 2 kp + 1 halves
                ldsm4<false>(b0, row + 16 * np * stride + 32 * kp + 8 * sel);
                ldsm4<false>(b1, row + (16 * np + 8) * stride + 32 * kp + 8 * sel);
                mma(d[0], a[2 * kp], b0[0], b0[1]);
                mma(d[1], a[2 * kp], b1[0], b1[1]);
                mma(d[0], a[2 * kp + 1], b0[2], b0[3]);
                mma(d[1], a[2 * kp + 1], b1[2], b1[3]);
            }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            out[np][2 * j] = pack2(fmaxf(d[j][0], 0.f), fmaxf(d[j][1], 0.f));
            out[np][2 * j + 1] = pack2(fmaxf(d[j][2], 0.f), fmaxf(d[j][3], 0.f));
        }
    }
}

__device__ __forceinline__ void output_layer(const uint32_t (*a)[4], const Image& s, int lane, float* d) {
    const int t = lane & 3;
    const float2 bb = *reinterpret_cast<const float2*>(s.b4 + 2 * t);
    d[0] = bb.x; d[1] = bb.y; d[2] = bb.x; d[3] = bb.y;
#pragma unroll
    for (int kp = 0; kp < 2; ++kp) {
        uint32_t b[4];
        ldsm4<false>(b, s.wt4 + (lane & 7) * kS64 + 32 * kp + 8 * (lane >> 3));
        mma(d, a[2 * kp], b[0], b[1]);
        mma(d, a[2 * kp + 1], b[2], b[3]);
    }
}

// Inference is bound by the layer chain as well (a 16-row tile is 76 MMAs in
// four dependent layers; the rows are 2 MB of traffic in 192k): 16 warps an SM
// with the weights fetched once per block.
constexpr int kFwdWarps = 8;
__global__ void __launch_bounds__(32 * kFwdWarps) forward_kernel(const Image* __restrict__ I,
                                                                 const float* __restrict__ X, int64_t n, int no,
                                                                 float* __restrict__ Y) {
    __shared__ Image s;
    dev::pdl_wait();
    fetch_image(&s, I);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int64_t tiles = (n + 15) / 16;
    for (int64_t tile = (int64_t)blockIdx.x * kFwdWarps + warp; tile < tiles; tile += (int64_t)gridDim.x * kFwdWarps) {
        const int64_t row0 = tile * 16;
        uint32_t a1[1][4], a2[4][4], a3[4][4], a4[4][4];
        float xv[8];
        read_x(X, row0 + g < n ? row0 + g : -1, row0 + g + 8 < n ? row0 + g + 8 : -1, t, xv);
        pack_x(xv, a1[0]);
        hidden_layer<1>(a1, s.wt1, kS16, s.b1, lane, a2);
        hidden_layer<4>(a2, s.wt2, kS64, s.b2, lane, a3);
        hidden_layer<4>(a3, s.wt3, kS64, s.b3, lane, a4);
        float d[4];
        output_layer(a4, s, lane, d);
        // this lane holds output columns 2t, 2t + 1 of rows g, g + 8
        const int c0 = 2 * t, c1 = 2 * t + 1;
        if (row0 + g < n) {
            if (c0 < no) Y[(row0 + g) * no + c0] = d[0];
            if (c1 < no) Y[(row0 + g) * no + c1] = d[1];
        }
        if (row0 + g + 8 < n) {
            if (c0 < no) Y[(row0 + g + 8) * no + c0] = d[2];
            if (c1 < no) Y[(row0 + g + 8) * no + c1] = d[3];
        }
    }
}

// ------------------------------------------------------------ gradients
constexpr int kGradWarps = 8;
constexpr int kRound = 16 * kGradWarps;  // rows of a block's round

struct GradSmem {
    Image w;
    // the round's layer inputs and errors, [row][feature]
    __nv_bfloat16 h0[kRound * kS16];
    __nv_bfloat16 h[3][kRound * kS64];
    __nv_bfloat16 dz[3][kRound * kS64];
    __nv_bfloat16 dy[kRound * 8];
    double loss[kGradWarps];
};

// store a warp's [16 rows x 64] A fragments row-major
__device__ __forceinline__ void stage(__nv_bfloat16* dst, const uint32_t (*a)[4], int rbase, int lane) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int kt = 0; kt < 4; ++kt)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            *reinterpret_cast<uint32_t*>(dst + (rbase + g + 8 * (q & 1)) * kS64 + 16 * kt + 8 * (q >> 1) + 2 * t) =
                a[kt][q];
}

// dZ of the layer below: (dz W^T) where the activation h is positive, rounded
// and packed; KT k-tiles over the layer's outputs (KT = 0: the output layer,
// whose 8 padded outputs fill half a k-tile).  W^T comes from the forward rows
// [out][in] by transposing loads.
template <int KT>
__device__ __forceinline__ void back_layer(const uint32_t (*dz)[4], const __nv_bfloat16* wt, const uint32_t (*h)[4],
                                           int lane, uint32_t (*out)[4]) {
    const __nv_bfloat16* row = wt + (lane & 7) * kS64;
    const int sel = lane >> 3;
#pragma unroll
    for (int np = 0; np < 4; ++np) {
        float d[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
        if (KT == 0) {
            uint32_t b[4];  // rows 0..7 of n-tiles 2 np, 2 np + 1 (the upper two matrices are not used)
            ldsm4<true>(b, row + 16 * np + 8 * (sel & 1));
            mma(d[0], dz[0], b[0], 0u);
            mma(d[1], dz[0], b[1], 0u);
        } else {
#pragma unroll
            for (int kt = 0; kt < KT; ++kt) {
                uint32_t b[4];  // n-tile 2 np rows 0..7, 8..15 of the k-tile; n-tile 2 np + 1 likewise
                ldsm4<true>(b, row + (16 * kt + 8 * (sel & 1)) * kS64 + 16 * np + 8 * (sel >> 1));
                mma(d[0], dz[kt], b[0], b[1]);
                mma(d[1], dz[kt], b[2], b[3]);
            }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int r = 0; r < 2; ++r) {  // rows g, g + 8
                const __nv_bfloat162 hv = *reinterpret_cast<const __nv_bfloat162*>(&h[np][2 * j + r]);
                out[np][2 * j + r] = pack2(__low2float(hv) > 0.f ? d[j][2 * r] : 0.f,
                                           __high2float(hv) > 0.f ? d[j][2 * r + 1] : 0.f);
            }
    }
}

// A fragment (16 features from f0 x 16 rows from r0) of H^T, H [row][feature]
__device__ __forceinline__ void frag_ht(uint32_t* a, const __nv_bfloat16* h, int stride, int r0, int f0, int lane) {
    ldsm4<true>(a, h + (r0 + (lane & 7) + 8 * (lane >> 4)) * stride + f0 + 8 * ((lane >> 3) & 1));
}
// B fragments (16 rows from r0 x outputs c0 .. c0 + 15) of dZ [row][out]: b[0..1] and b[2..3]
__device__ __forceinline__ void frag_dz(uint32_t* b, const __nv_bfloat16* z, int r0, int c0, int lane) {
    ldsm4<true>(b, z + (r0 + (lane & 7) + 8 * ((lane >> 3) & 1)) * kS64 + c0 + 8 * (lane >> 4));
}

// n rows of the minibatch, drawn from n_data rows of (X, T) by data_row.  Warp
// w owns of dW2 and dW3 feature rows 16 (w % 4) .. + 15, outputs 32 (w / 4) ..
// + 31; of dW1 outputs 8 w .. + 7; warps 0..3 of dW4 feature rows 16 w .. + 15.
__global__ void __launch_bounds__(32 * kGradWarps, 1)
    grad_kernel(const Image* __restrict__ I, const float* __restrict__ X, const float* __restrict__ T, int no, int64_t n,
                int64_t n_data, uint64_t seed, uint64_t step, float inv_n2, float* __restrict__ partial,
                double* __restrict__ loss_partial) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    GradSmem& s = *reinterpret_cast<GradSmem*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    dev::pdl_trigger();
    float m1[4] = {}, m2[4][4] = {}, m3[4][4] = {}, m4[4] = {};
    float mb0 = 0.f, mb1 = 0.f;
    double my_loss = 0.0;
    // contiguous 16-row tiles per block
    const int64_t tiles = (n + 15) / 16;
    const int64_t tile0 = tiles * blockIdx.x / gridDim.x, tile1 = tiles * (blockIdx.x + 1) / gridDim.x;
    // the warp's 16 rows of the round at tb: drawn and read a round ahead, so
    // that the draw and the latency of scattered rows lie behind other work
    float xv[8], tv[4];
    bool real[2];
    auto read_rows = [&](int64_t tb) {
        const int64_t row0 = (tb + warp) * 16;
        int64_t mine = -1;
        if (tb + warp < tile1 && lane < 16 && row0 + lane < n) mine = data_row(row0 + lane, n_data, seed, step);
        const int64_t src0 = __shfl_sync(0xffffffffu, mine, g), src1 = __shfl_sync(0xffffffffu, mine, g + 8);
        read_x(X, src0, src1, t, xv);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int c = 2 * t + (q & 1);
            const int64_t src = q < 2 ? src0 : src1;
            tv[q] = c < no && src >= 0 ? T[src * no + c] : 0.f;
        }
        real[0] = src0 >= 0;
        real[1] = src1 >= 0;
    };
    // the data are the caller's, complete before the first launch of the call,
    // which is an ordinary one; the image is written by the kernel before
    read_rows(tile0);
    dev::pdl_wait();
    fetch_image(&s.w, I);
    for (int64_t tb = tile0; tb < tile1; tb += kGradWarps) {
        const int act = (int)(tile1 - tb < kGradWarps ? tile1 - tb : kGradWarps);  // tiles of this round
        const int rb = warp * 16;
        if (warp < act) {
            // ---- forward for the warp's 16 rows, keeping every activation
            uint32_t a1[1][4], a2[4][4], a3[4][4], a4[4][4];
            pack_x(xv, a1[0]);
            hidden_layer<1>(a1, s.w.wt1, kS16, s.w.b1, lane, a2);
            hidden_layer<4>(a2, s.w.wt2, kS64, s.w.b2, lane, a3);
            hidden_layer<4>(a3, s.w.wt3, kS64, s.w.b3, lane, a4);
            float y[4];
            output_layer(a4, s.w, lane, y);
            // ---- output error dY = 2 (Y - T) / n (zero on padding rows and
            // columns); this lane holds columns 2t, 2t + 1 of rows g, g + 8
            float dy[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int c = 2 * t + (q & 1);
                if (c < no && real[q >> 1]) {
                    const float e = y[q] - tv[q];
                    my_loss += (double)e * e;
                    dy[q] = inv_n2 * e;
                }
            }
            uint32_t ady[1][4] = {{pack2(dy[0], dy[1]), pack2(dy[2], dy[3]), 0u, 0u}};
            // ---- the inputs of every layer and dY
#pragma unroll
            for (int q = 0; q < 4; ++q)
                *reinterpret_cast<uint32_t*>(s.h0 + (rb + g + 8 * (q & 1)) * kS16 + 8 * (q >> 1) + 2 * t) = a1[0][q];
            stage(s.h[0], a2, rb, lane);
            stage(s.h[1], a3, rb, lane);
            stage(s.h[2], a4, rb, lane);
            *reinterpret_cast<uint32_t*>(s.dy + (rb + g) * 8 + 2 * t) = ady[0][0];
            *reinterpret_cast<uint32_t*>(s.dy + (rb + g + 8) * 8 + 2 * t) = ady[0][1];
            // ---- back through the layers: dZ3 = (dY W4^T) * [H3 > 0], ...
            uint32_t dz[4][4], dn[4][4];
            back_layer<0>(ady, s.w.wt4, a4, lane, dz);
            stage(s.dz[2], dz, rb, lane);
            back_layer<4>(dz, s.w.wt3, a3, lane, dn);
            stage(s.dz[1], dn, rb, lane);
            back_layer<4>(dn, s.w.wt2, a2, lane, dz);
            stage(s.dz[0], dz, rb, lane);
        }
        if (tb + kGradWarps < tile1) read_rows(tb + kGradWarps);
        __syncthreads();
        // ---- weight gradients: chains of up to 64 rows, added in FP32
        const int mt = warp & 3, c0 = 32 * (warp >> 2);
        for (int half = 0; 4 * half < act; ++half) {
            float d1[4] = {}, d2[4][4] = {}, d3[4][4] = {}, d4[4] = {};
            const int kend = act < 4 * half + 4 ? act : 4 * half + 4;
            for (int kt = 4 * half; kt < kend; ++kt) {
                const int r0 = 16 * kt;
                uint32_t a[4], b[8];
                frag_ht(a, s.h[0], kS64, r0, 16 * mt, lane);
                frag_dz(b, s.dz[1], r0, c0, lane);
                frag_dz(b + 4, s.dz[1], r0, c0 + 16, lane);
#pragma unroll
                for (int j = 0; j < 4; ++j) mma(d2[j], a, b[2 * j], b[2 * j + 1]);
                frag_ht(a, s.h[1], kS64, r0, 16 * mt, lane);
                frag_dz(b, s.dz[2], r0, c0, lane);
                frag_dz(b + 4, s.dz[2], r0, c0 + 16, lane);
#pragma unroll
                for (int j = 0; j < 4; ++j) mma(d3[j], a, b[2 * j], b[2 * j + 1]);
                frag_ht(a, s.h0, kS16, r0, 0, lane);
                frag_dz(b, s.dz[0], r0, 16 * (warp >> 1), lane);
                mma(d1, a, warp & 1 ? b[2] : b[0], warp & 1 ? b[3] : b[1]);
                if (warp < 4) {
                    frag_ht(a, s.h[2], kS64, r0, 16 * warp, lane);
                    // rows 0..7 and 8..15 of dY (lanes above 15 repeat them)
                    ldsm4<true>(b, s.dy + (r0 + (lane & 7) + 8 * ((lane >> 3) & 1)) * 8);
                    mma(d4, a, b[0], b[1]);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                m1[i] += d1[i];
                m4[i] += d4[i];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    m2[j][i] += d2[j][i];
                    m3[j][i] += d3[j][i];
                }
            }
        }
        // ---- bias gradients: sums of the BF16 errors over the round's rows;
        // threads 0..191 take column pairs (even and odd rows apart), 192.. dY
        if (threadIdx.x < 192) {
            const int pr = threadIdx.x >> 1, layer = pr >> 5, c = 2 * (pr & 31);
            float u = 0.f, v = 0.f;
            for (int r = threadIdx.x & 1; r < 16 * act; r += 2) {
                const __nv_bfloat162 z = *reinterpret_cast<const __nv_bfloat162*>(s.dz[layer] + r * kS64 + c);
                u += __low2float(z);
                v += __high2float(z);
            }
            mb0 += u;
            mb1 += v;
        } else if (threadIdx.x < 192 + 8) {
            float u = 0.f;
            for (int r = 0; r < 16 * act; ++r) u += __bfloat162float(s.dy[r * 8 + threadIdx.x - 192]);
            mb0 += u;
        }
        __syncthreads();
    }
    // ---- loss of the block (fixed order), then the block's partial gradient
    for (int o = 16; o > 0; o >>= 1) my_loss += __shfl_xor_sync(0xffffffffu, my_loss, o);
    if (lane == 0) s.loss[warp] = my_loss;
    __syncthreads();
    if (threadIdx.x == 0) {
        double l = 0.0;
        for (int w = 0; w < kGradWarps; ++w) l += s.loss[w];
        loss_partial[blockIdx.x] = l;
    }
    float* out = partial + (size_t)blockIdx.x * param_count(no);
    auto put = [&](int o, int ld, int r, int c, const float* v) {  // C fragment at row r, column c
        out[o + r * ld + c] = v[0];
        out[o + r * ld + c + 1] = v[1];
        out[o + (r + 8) * ld + c] = v[2];
        out[o + (r + 8) * ld + c + 1] = v[3];
    };
    const int mt = warp & 3, c0 = 32 * (warp >> 2);
    put(oW1, kH, g, 8 * warp + 2 * t, m1);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        put(oW2, kH, 16 * mt + g, c0 + 8 * j + 2 * t, m2[j]);
        put(oW3, kH, 16 * mt + g, c0 + 8 * j + 2 * t, m3[j]);
    }
    if (warp < 4)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (2 * t + (i & 1) < no) out[oW4 + (16 * warp + g + 8 * (i >> 1)) * no + 2 * t + (i & 1)] = m4[i];
    // even and odd rows of a bias column together
    mb0 += __shfl_down_sync(0xffffffffu, threadIdx.x < 192 ? mb0 : 0.f, 1);
    mb1 += __shfl_down_sync(0xffffffffu, mb1, 1);
    if (threadIdx.x < 192) {
        if (!(threadIdx.x & 1)) {
            const int pr = threadIdx.x >> 1, layer = pr >> 5, c = 2 * (pr & 31);
            const int o = layer == 0 ? oB1 : (layer == 1 ? oB2 : oB3);
            out[o + c] = mb0;
            out[o + c + 1] = mb1;
        }
    } else if ((int)threadIdx.x < 192 + no) {
        out[off_b4(no) + threadIdx.x - 192] = mb0;
    }
}

// Adds the blocks' partial gradients and losses in a fixed order (eight slices
// of the blocks per parameter side by side, then the slices), and with ADAM
// takes the bias-corrected Adam step (Kingma & Ba) on the FP32 master
// parameters and writes the changed weights into the image.  It is bound by
// reading the partials (38 KB a block) from L2, so it spreads each parameter
// over eight threads.
constexpr int kSumParams = 32, kSumSlices = 8;
template <bool ADAM>
__global__ void __launch_bounds__(kSumParams * kSumSlices)
    sum_partials(int nb, int kp, int no, const float* __restrict__ partial, const double* __restrict__ loss_partial,
                 float* __restrict__ grad, double* __restrict__ loss, float* __restrict__ p, float* __restrict__ m,
                 float* __restrict__ v, Image* __restrict__ I, float lr, float b1, float b2, float eps, float c1,
                 float c2) {
    __shared__ float slice[kSumSlices][kSumParams];
    const int lane = threadIdx.x % kSumParams, sl = threadIdx.x / kSumParams;
    const int i = blockIdx.x * kSumParams + lane;
    dev::pdl_trigger();
    dev::pdl_wait();
    float acc = 0.f;
    if (i < kp)
        for (int b = sl; b < nb; b += kSumSlices) acc += partial[(size_t)b * kp + i];
    slice[sl][lane] = acc;
    __syncthreads();
    if (sl == 0 && i < kp) {
        float gi = slice[0][lane];
#pragma unroll
        for (int q = 1; q < kSumSlices; ++q) gi += slice[q][lane];
        grad[i] = gi;
        if (ADAM) {
            const float mi = b1 * m[i] + (1.f - b1) * gi;
            const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
            m[i] = mi;
            v[i] = vi;
            const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
            p[i] = pi;
            image_put(I, no, i, pi);
        }
    }
    if (blockIdx.x == 0 && sl == 1) {  // one warp: 32 strided sums, then across the lanes
        double l = 0.0;
        for (int b = lane; b < nb; b += 32) l += loss_partial[b];
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) *loss = l;
    }
}

}  // namespace mlp
}  // namespace mlbm

using namespace mlbm;

struct mlbm_mlp {
    mlp::Image* img = nullptr;  // BF16 weights and biases, kept in line with p
    float* p = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    float* grad = nullptr;
    float* partial = nullptr;
    double* loss_partial = nullptr;
    double* loss = nullptr;
    int max_blocks = 0;
    int n_out = 2;
    int kp = 0;     // parameter count
    int64_t t = 0;  // Adam step count
};

namespace {
#define MLP_CUDA(call)                                                                                \
    do {                                                                                              \
        cudaError_t e_ = (call);                                                                      \
        if (e_ != cudaSuccess) return set_error(MLBM_E_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

uint64_t splitmix(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
double gauss(uint64_t& s) {
    const double u1 = ((splitmix(s) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    const double u2 = ((splitmix(s) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    return std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2);
}
constexpr int kMaxGradBlocks = 152;  // one per SM
int grad_blocks(int64_t n) {
    const int64_t rounds = (n + mlp::kRound - 1) / mlp::kRound;
    return (int)std::max<int64_t>(1, std::min<int64_t>(rounds, kMaxGradBlocks));
}
}  // namespace

extern "C" {

int64_t mlbm_mlp_param_count(int n_out) {
    return n_out >= 1 && n_out <= mlp::kMaxOut ? mlp::param_count(n_out) : -1;
}

int mlbm_mlp_outputs(const mlbm_mlp* m) { return m ? m->n_out : -1; }

mlbm_status mlbm_mlp_create(mlbm_mlp** out, int n_out, uint64_t seed) {
    clear_error();
    if (!out || n_out < 1 || n_out > mlp::kMaxOut) return set_error(MLBM_E_INVALID, "mlp_create: bad arguments");
    *out = nullptr;
    auto* m = new (std::nothrow) mlbm_mlp;
    if (!m) return set_error(MLBM_E_OOM, "mlp_create: out of host memory");
    m->max_blocks = kMaxGradBlocks;
    m->n_out = n_out;
    m->kp = mlp::param_count(n_out);
    cudaError_t e = cudaSuccess;
    e = e == cudaSuccess ? cudaMalloc(&m->img, sizeof(mlp::Image)) : e;
    e = e == cudaSuccess ? cudaMemset(m->img, 0, sizeof(mlp::Image)) : e;
    e = e == cudaSuccess ? cudaMalloc(&m->p, m->kp * 4) : e;
    e = e == cudaSuccess ? cudaMalloc(&m->m, m->kp * 4) : e;
    e = e == cudaSuccess ? cudaMalloc(&m->v, m->kp * 4) : e;
    e = e == cudaSuccess ? cudaMalloc(&m->grad, m->kp * 4) : e;
    e = e == cudaSuccess ? cudaMalloc(&m->partial, (size_t)m->max_blocks * m->kp * 4) : e;
    e = e == cudaSuccess ? cudaMalloc(&m->loss_partial, (size_t)m->max_blocks * 8) : e;
    e = e == cudaSuccess ? cudaMalloc(&m->loss, 8) : e;
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        mlbm_mlp_destroy(m);
        return set_error(MLBM_E_CUDA, std::string("mlp_create: ") + cudaGetErrorString(e));
    }
    // He-normal weights, zero biases
    std::vector<float> h(m->kp, 0.f);
    uint64_t st = seed * 0x2545F4914F6CDD1Dull + 1;
    const int sizes[5] = {mlp::kIn, mlp::kH, mlp::kH, mlp::kH, n_out};
    int o = 0;
    for (int l = 0; l < 4; ++l) {
        const double sd = std::sqrt(2.0 / sizes[l]);
        for (int i = 0; i < sizes[l] * sizes[l + 1]; ++i) h[o + i] = (float)(sd * gauss(st));
        o += sizes[l] * sizes[l + 1] + sizes[l + 1];
    }
    mlbm_status s = mlbm_mlp_set_params(m, h.data());
    if (s != MLBM_OK) {
        std::string msg = mlbm_last_error();
        mlbm_mlp_destroy(m);
        return set_error(s, msg);
    }
    *out = m;
    return MLBM_OK;
}

void mlbm_mlp_destroy(mlbm_mlp* m) {
    if (!m) return;
    cudaFree(m->img); cudaFree(m->p); cudaFree(m->m); cudaFree(m->v); cudaFree(m->grad); cudaFree(m->partial);
    cudaFree(m->loss_partial); cudaFree(m->loss);
    delete m;
}

mlbm_status mlbm_mlp_set_params(mlbm_mlp* m, const float* params) {
    if (!m || !params) return set_error(MLBM_E_INVALID, "mlp_set_params: NULL argument");
    MLP_CUDA(cudaMemcpy(m->p, params, m->kp * 4, cudaMemcpyHostToDevice));
    mlp::take_params<<<(m->kp + 255) / 256, 256>>>(m->kp, m->n_out, m->p, m->img, m->m, m->v);
    MLP_CUDA(cudaGetLastError());
    MLP_CUDA(cudaStreamSynchronize(nullptr));
    m->t = 0;
    return MLBM_OK;
}

mlbm_status mlbm_mlp_get_params(mlbm_mlp* m, float* params) {
    if (!m || !params) return set_error(MLBM_E_INVALID, "mlp_get_params: NULL argument");
    MLP_CUDA(cudaMemcpy(params, m->p, m->kp * 4, cudaMemcpyDeviceToHost));
    return MLBM_OK;
}

mlbm_status mlbm_mlp_forward_device(mlbm_mlp* m, const float* X, int64_t n, float* Y, void* stream) {
    if (!m || (n > 0 && (!X || !Y)) || n < 0) return set_error(MLBM_E_INVALID, "mlp_forward: bad arguments");
    if (n == 0) return MLBM_OK;
    const int64_t tiles = (n + 15) / 16;
    const int blocks =
        (int)std::max<int64_t>(1, std::min<int64_t>((tiles + mlp::kFwdWarps - 1) / mlp::kFwdWarps, 152 * 2));
    mlp::forward_kernel<<<blocks, 32 * mlp::kFwdWarps, 0, static_cast<cudaStream_t>(stream)>>>(m->img, X, n, m->n_out,
                                                                                               Y);
    MLP_CUDA(cudaGetLastError());
    return MLBM_OK;
}

}  // extern "C"

namespace {
// one gradient evaluation over n minibatch rows into m->grad and the device
// loss sum m->loss, and with lr > 0 the Adam step number m->t on it
mlbm_status grad_pass(mlbm_mlp* m, const float* X, const float* T, int64_t n, int64_t n_data, uint64_t seed,
                      uint64_t step, float lr, bool first, cudaStream_t st) {
    const int nb = grad_blocks(n);
    const size_t smem = sizeof(mlp::GradSmem);
    MLP_CUDA(cudaFuncSetAttribute(mlp::grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const float inv_n2 = (float)(2.0 / (double)n);
    if (first) {  // reads the caller's data at once, so not before what is on the stream has ended
        mlp::grad_kernel<<<nb, 32 * mlp::kGradWarps, smem, st>>>(m->img, X, T, m->n_out, n, n_data, seed, step, inv_n2,
                                                                 m->partial, m->loss_partial);
        MLP_CUDA(cudaGetLastError());
    } else {
        MLP_CUDA(launch_pdl_smem(mlp::grad_kernel, nb, 32 * mlp::kGradWarps, smem, st, m->img, X, T, m->n_out, n,
                                 n_data, seed, step, inv_n2, m->partial, m->loss_partial));
    }
    const int blocks = (m->kp + mlp::kSumParams - 1) / mlp::kSumParams, threads = mlp::kSumParams * mlp::kSumSlices;
    const double c1 = 1.0 - std::pow(0.9, (double)m->t), c2 = 1.0 - std::pow(0.999, (double)m->t);
    auto fn = lr > 0 ? mlp::sum_partials<true> : mlp::sum_partials<false>;
    MLP_CUDA(launch_pdl_smem(fn, blocks, threads, 0, st, nb, m->kp, m->n_out, m->partial, m->loss_partial, m->grad,
                             m->loss, m->p, m->m, m->v, m->img, lr, 0.9f, 0.999f, 1e-8f, (float)c1, (float)c2));
    return MLBM_OK;
}

mlbm_status read_loss(mlbm_mlp* m, int64_t n, double* loss, cudaStream_t st) {
    double h = 0;
    MLP_CUDA(cudaMemcpyAsync(&h, m->loss, 8, cudaMemcpyDeviceToHost, st));
    MLP_CUDA(cudaStreamSynchronize(st));
    *loss = h / (double)n;
    return MLBM_OK;
}
}  // namespace

extern "C" {

mlbm_status mlbm_mlp_gradients_device(mlbm_mlp* m, const float* X, const float* T, int64_t n, float* grads,
                                      double* loss, void* stream) {
    if (!m || !X || !T || n <= 0) return set_error(MLBM_E_INVALID, "mlp_gradients: bad arguments");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    mlbm_status s = grad_pass(m, X, T, n, n, 0, 0, 0.f, true, st);
    if (s != MLBM_OK) return s;
    if (grads) MLP_CUDA(cudaMemcpyAsync(grads, m->grad, m->kp * 4, cudaMemcpyDeviceToDevice, st));
    if (loss) return read_loss(m, n, loss, st);
    return MLBM_OK;
}

mlbm_status mlbm_mlp_train_device(mlbm_mlp* m, const float* X, const float* T, int64_t n, int64_t batch,
                                  int64_t steps, float lr, uint64_t seed, double* loss, void* stream) {
    if (!m || !X || !T || n <= 0 || batch <= 0 || steps < 0 || !(lr > 0) || (seed == 0 && batch != n))
        return set_error(MLBM_E_INVALID, "mlp_train: bad arguments");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    for (int64_t k = 0; k < steps; ++k) {
        const uint64_t draw = (uint64_t)m->t;
        m->t += 1;
        mlbm_status s = grad_pass(m, X, T, batch, n, seed, draw, lr, k == 0, st);
        if (s != MLBM_OK) {
            m->t -= 1;
            return s;
        }
    }
    if (loss) {
        if (steps == 0) return set_error(MLBM_E_INVALID, "mlp_train: no step taken, no loss to report");
        return read_loss(m, batch, loss, st);
    }
    return MLBM_OK;
}

}  // extern "C"
