// Area-weighted sums of FP32 fields with FP64 results, formed on the FP32 pipe.
//
// This GPU issues two FP64 instructions per clock and SM, so the six sums of a
// node (four conversions, a square root, six accumulations: ~25 instructions)
// took 12 clocks a node, 523 us for 13.25M nodes whose 225 MB need 33 us.
// Here every sum is three FP32 numbers of falling magnitude, fed by error-free
// transforms (Knuth's TwoSum, the FMA product error; the square root by two
// correction steps on its exact residual), so what is lost per node lies
// 2^-68 below it, and the three are added into FP64 every kFlush nodes:
// fewer FP64 roundings than one per node.  For that every product and error
// term has to lie in the FP32 range: a node takes the FP64 path when a value is
// neither zero nor within [2^-45, 2^45] (u^2 and rho A then reach 2^90, and
// their last bits 2^-136), when |u|^2 A, the one product of three values, is
// neither zero nor within [2^-77, 2^110] (at the lower end the third of its
// parts rounds at 2^-149, 2^-72 of it; kFlush terms at the upper end add up to
// 2^118), and for infinities and NaN.  13.25M nodes: 523 -> 144 us.  Blocks of
// one or two nodes a thread keep to FP64, whose pipe they do not fill, and skip
// the flush (us a call, FP64 / FP32 pipe: 64 nodes 8.9 / 10.4, 256 10.0 / 11.4,
// 512 11.6 / 12.1; FP64 alone at 600 12.5 / 12.3, at 1000 17.0 / 13.7).
#pragma once

#include <cuda_runtime.h>

namespace mlbm {
namespace dev {

__device__ __forceinline__ void exact_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void exact_prod(float a, float b, float& p, float& e) {
    p = __fmul_rn(a, b);
    e = __fmaf_rn(a, b, -p);
}

// a running sum h + m + l
struct Float3Sum {
    float h = 0.f, m = 0.f, l = 0.f;
    __device__ __forceinline__ void add(float x) {
        float e, f;
        exact_sum(h, x, h, e);
        exact_sum(m, e, m, f);
        l += f;
    }
    __device__ __forceinline__ void add_low(float x) {  // a term ~2^-24 of the sum's
        float f;
        exact_sum(m, x, m, f);
        l += f;
    }
    __device__ __forceinline__ void add_prod(float a, float b) {
        float p, e;
        exact_prod(a, b, p, e);
        add(p);
        add_low(e);
    }
    // (x0 + x1 + x2) a, the terms of falling magnitude
    __device__ __forceinline__ void add_prod3(float x0, float x1, float x2, float a) {
        float p, e, q, f;
        exact_prod(x0, a, p, e);
        exact_prod(x1, a, q, f);
        add(p);
        add_low(e);
        add_low(q);
        l += __fmaf_rn(x2, a, f);
    }
    __device__ __forceinline__ void flush(double& s) {
        s += (double)h + ((double)m + (double)l);
        h = m = l = 0.f;
    }
};

// sums of A, rho A, ux A, uy A, |u| A, |u|^2 A
struct FieldSums {
    static constexpr int kFlush = 256;
    static constexpr int kFew = 2;  // nodes a thread up to which add64 is the faster one
    static constexpr float kLeast = 6.617444900424222e-24f, kMost = 1.298074214633707e33f;  // 2^-77, 2^110
    Float3Sum f[6];
    double s[6] = {0, 0, 0, 0, 0, 0};
    int held = 0;

    static __device__ __forceinline__ bool plain(float x) {
        const float a = fabsf(x);
        return x == 0.f || (a >= 2.84217094304040074e-14f && a <= 3.5184372088832e13f);
    }
    __device__ __forceinline__ void add64(float rho, float u, float v, float a) {
        const double da = a, du = u, dv = v, m2 = du * du + dv * dv;
        s[0] += da;
        s[1] += (double)rho * da;
        s[2] += du * da;
        s[3] += dv * da;
        s[4] += sqrt(m2) * da;
        s[5] += m2 * da;
    }
    __device__ __forceinline__ void add(float rho, float u, float v, float a) {
        // |u|^2 = p + e + q + g, and x0 its leading part
        float p, e, q, g, x0, x1, x2, t, w;
        exact_prod(u, u, p, e);
        exact_prod(v, v, q, g);
        exact_sum(p, q, x0, t);
        const float m2a = fabsf(__fmul_rn(x0, a));
        if (!(plain(rho) && plain(u) && plain(v) && plain(a) && (m2a == 0.f || (m2a >= kLeast && m2a <= kMost)))) {
            add64(rho, u, v, a);
            return;
        }
        f[0].add(a);
        f[1].add_prod(rho, a);
        f[2].add_prod(u, a);
        f[3].add_prod(v, a);
        // |u|^2 = x0 + x1 + x2
        exact_sum(e, g, x1, x2);
        exact_sum(t, x1, x1, w);
        x2 += w;
        exact_sum(x0, x1, x0, x1);
        f[5].add_prod3(x0, x1, x2, a);
        // |u| = r0 + r1 + r2: r1 and r2 from the residual |u|^2 - (r0 + ...)^2
        float r0 = __fsqrt_rn(x0), r1 = 0.f, r2 = 0.f;
        if (r0 > 0.f) {
            const float half = __fdividef(0.5f, r0);
            exact_prod(r0, r0, p, e);
            float d0 = __fsub_rn(x0, p), d1;  // exact: x0 and p are within a few ulp
            exact_sum(x1, -e, t, w);
            exact_sum(d0, t, d0, d1);
            d1 += w + x2;
            r1 = (d0 + d1) * half;
            exact_prod(2.f * r0, r1, p, e);
            r2 = ((__fsub_rn(d0, p) - e) + (d1 - r1 * r1)) * half;
        }
        f[4].add_prod3(r0, r1, r2, a);
        if (++held == kFlush) flush();
    }
    __device__ __forceinline__ void flush() {
        if (!held) return;
#pragma unroll
        for (int q = 0; q < 6; ++q) f[q].flush(s[q]);
        held = 0;
    }
};

}  // namespace dev
}  // namespace mlbm
