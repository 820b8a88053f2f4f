// State I/O, macroscopic fields, the momentum-exchange force and the FP64
// reductions; the step kernels are in kernels_bgk.cu, kernels_tau1.cu,
// kernels_rbf.cu, kernels_warp.cu and kernels_tma.cu.
//
// All population values are stored minus their weight omega_k (and rho as
// rho - 1) so that FP32 keeps the small deviations that carry the flow.
#include <cstdio>

#include "device_common.cuh"
#include "float_sums.cuh"
#include "kernels.h"
#include "launch_util.cuh"

namespace mlbm {
namespace dev {

// ------------------------------------------------------------- state I/O
__global__ void set_bgk_from_f64(int n, const int* __restrict__ perm, const double* __restrict__ f,
                                 float4* __restrict__ f8, float* __restrict__ f0) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const double* fi = f + 9 * (size_t)perm[p];
    float g[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const double w = k == 0 ? 4.0 / 9.0 : (k <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
        g[k] = (float)(fi[k] - w);
    }
    f8[2 * (size_t)p] = make_float4(g[1], g[2], g[3], g[4]);
    f8[2 * (size_t)p + 1] = make_float4(g[5], g[6], g[7], g[8]);
    f0[p] = g[0];
}

__global__ void get_bgk_to_f64(int n, const int* __restrict__ perm, const float4* __restrict__ f8,
                               const float* __restrict__ f0, double* __restrict__ f) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    double* fi = f + 9 * (size_t)perm[p];
    const float4 a = f8[2 * (size_t)p], b = f8[2 * (size_t)p + 1];
    const float g[9] = {f0[p], a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const double w = k == 0 ? 4.0 / 9.0 : (k <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
        fi[k] = (double)g[k] + w;
    }
}

// state at t = 0 from (rho, u): BGK populations at equilibrium, computed in FP64
__global__ void set_bgk_equilibrium(int n, const int* __restrict__ perm, const double* __restrict__ ru,
                                    float4* __restrict__ f8, float* __restrict__ f0) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const double* v = ru + 3 * (size_t)perm[p];
    const double rho = v[0], ux = v[1], uy = v[2];
    const double usq = ux * ux + uy * uy;
    float g[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const double w = k == 0 ? 4.0 / 9.0 : (k <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
        const double eu = ex_of(k) * ux + ey_of(k) * uy;
        g[k] = (float)(w * ((rho - 1.0) + rho * (3.0 * eu + 4.5 * eu * eu - 1.5 * usq)));
    }
    f8[2 * (size_t)p] = make_float4(g[1], g[2], g[3], g[4]);
    f8[2 * (size_t)p + 1] = make_float4(g[5], g[6], g[7], g[8]);
    f0[p] = g[0];
}

__global__ void set_tau1_from_f64(int n, const int* __restrict__ perm, const double* __restrict__ ru,
                                  float4* __restrict__ s) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const double* v = ru + 3 * (size_t)perm[p];
    s[p] = make_float4((float)(v[0] - 1.0), (float)v[1], (float)v[2], 0.f);
}

// (rho - 1, ux, uy) of a BGK state: rho = sum f, rho u = sum f e - rho a / 2
__device__ __forceinline__ void bgk_moments(const float4& a, const float4& b, float g0, float ax, float ay, float& dr,
                                            float& ux, float& uy) {
    dr = g0 + (a.x + a.y + a.z + a.w) + (b.x + b.y + b.z + b.w);
    const float jx = (a.x - a.z) + (b.x - b.y) + (b.w - b.z);
    const float jy = (a.y - a.w) + (b.x + b.y) - (b.z + b.w);
    const float rho = 1.0f + dr;
    ux = jx / rho - 0.5f * ax;
    uy = jy / rho - 0.5f * ay;
}

// (rho, ux, uy) of caller's node i of n into FP64 caller-order arrays: rows
// [n][3], or (split) rho[n] followed by u[n][2]
__device__ __forceinline__ void put_fields(double* out, int split, int n, int i, double rho, float ux, float uy) {
    double* r = split ? out + i : out + 3 * (size_t)i;
    double* u = split ? out + (size_t)n + 2 * (size_t)i : r + 1;
    r[0] = rho;
    u[0] = ux;
    u[1] = uy;
}

// rho, u of the state into FP64 caller-order arrays
__global__ void macroscopics_bgk(int n, const int* __restrict__ perm, const float4* __restrict__ f8,
                                 const float* __restrict__ f0, float ax0, float ay0,
                                 const uint16_t* __restrict__ node_sample, const Collide* __restrict__ coll, int split,
                                 double* __restrict__ out) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const float ax = node_sample ? coll[node_sample[p]].ax : ax0;
    const float ay = node_sample ? coll[node_sample[p]].ay : ay0;
    float dr, ux, uy;
    bgk_moments(f8[2 * (size_t)p], f8[2 * (size_t)p + 1], f0[p], ax, ay, dr, ux, uy);
    put_fields(out, split, n, perm[p], 1.0 + (double)dr, ux, uy);
}

__global__ void macroscopics_tau1(int n, const int* __restrict__ perm, const float4* __restrict__ s, int split,
                                  double* __restrict__ out) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const float4 a = s[p];
    put_fields(out, split, n, perm[p], 1.0 + (double)a.x, a.y, a.z);
}

// --------------------------------------------------------- wall force
// Momentum handed to the solids in the next streaming step: sum over links of
// 2 (f_k(t+1, x) - omega_k) e_{k'} area_x / s^2 (relative to the rest state,
// whose uniform pressure exerts no net force on a closed body), per-block
// FP64 partials added in a fixed order.
template <int KQ>
__global__ void __launch_bounds__(128) force_kernel(Stencil S, int model, int n_link_nodes,
                                                    const int* __restrict__ link_nodes,
                                                    const float* __restrict__ area_over_s2,
                                                    const float4* __restrict__ st8, const float4* __restrict__ ruv,
                                                    Collide C, double* __restrict__ partial) {
    double fx = 0.0, fy = 0.0;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n_link_nodes; e += gridDim.x * blockDim.x) {
        const int p = link_nodes[e];
        const Collide Cn = collide_of(S, C, p);
        const uint8_t meta = S.meta[p];
        const int kind = meta & 3;
        const LinkRec L = S.links[S.link_slot[p]];
        const float r = (kind == 1) ? S.lag_r[p] : 0.f;
        const float cx = (kind == 1) ? (float)ex_of(meta >> 4) : 0.f;
        const float cy = (kind == 1) ? (float)ey_of(meta >> 4) : 0.f;
        const double a = area_over_s2[p];
        for (int k = 1; k < 9; ++k) {
            if (!((L.mask >> k) & 1u)) continue;
            const int kp = opp_of(k);
            float val;
            if (model == 0) {
                if (S.bb_mode == 0) {
                    val = pop(st8, p, kp);
                } else if (kind == 0 && !S.rec) {
                    val = rbf_general<KQ>(S, st8, p, k - 1, kp);
                } else if (kind == 0) {
                    float pb[6];
                    basis_at(k, L.t[k - 1], pb);
                    val = wls_general<KQ>(S, st8, p, kp, pb);
                } else {
                    int ids[9];
                    lag_block(S, p, ids);
                    float lx[3], ly[3];
                    lag3(L.t[k - 1] * r * ex_of(k) - cx, lx[0], lx[1], lx[2]);
                    lag3(L.t[k - 1] * r * ey_of(k) - cy, ly[0], ly[1], ly[2]);
                    val = 0.f;
                    for (int b = 0; b < 3; ++b)
                        for (int aa = 0; aa < 3; ++aa) val = fmaf(lx[aa] * ly[b], pop(st8, ids[b * 3 + aa], kp), val);
                }
            } else {
                float d[3];
                if (S.bb_mode == 0) {
                    const float4 me = ruv[p];
                    d[0] = me.x; d[1] = me.y; d[2] = me.z;
                } else if (kind == 0 && !S.rec) {
                    d[0] = d[1] = d[2] = 0.f;
                    for (int q = 0; q < KQ; ++q) {
                        const int4 id = S.idx[(size_t)q * S.n_pad + p];
                        const float4 wq = S.Wr[(size_t)((k - 1) * KQ + q) * S.n_pad + p];
                        const int ids[4] = {id.x, id.y, id.z, id.w};
                        const float ws[4] = {wq.x, wq.y, wq.z, wq.w};
                        for (int cq = 0; cq < 4; ++cq) {
                            const float4 v = ruv[ids[cq]];
                            d[0] = fmaf(ws[cq], v.x, d[0]);
                            d[1] = fmaf(ws[cq], v.y, d[1]);
                            d[2] = fmaf(ws[cq], v.z, d[2]);
                        }
                    }
                } else if (kind == 0) {
                    float pb[6];
                    basis_at(k, L.t[k - 1], pb);
                    d[0] = d[1] = d[2] = 0.f;
                    // centred on the node's own values, as its own column is not stored
                    const float4* lane_rows = rec_lane<KQ>(S, p);
                    const float4 me = ruv[p];
                    for (int q = 0; q < KQ; ++q) {
                        const int4 id = rec_ids<KQ>(lane_rows, q, p, LdCached{});
                        float4 m[6];
                        rec_group<KQ>(lane_rows, q, m, LdCached{});
                        const int ids[4] = {id.x, id.y, id.z, id.w};
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            float tcol[6], mm[6];
#pragma unroll
                            for (int aa = 0; aa < 6; ++aa) tcol[aa] = reinterpret_cast<const float*>(m)[4 * aa + c];
                            unbasis(tcol, mm);
                            float w = 0.f;
#pragma unroll
                            for (int aa = 0; aa < 6; ++aa) w = fmaf(pb[aa], mm[aa], w);
                            const float4 v = ruv[ids[c]];
                            d[0] = fmaf(w, v.x - me.x, d[0]);
                            d[1] = fmaf(w, v.y - me.y, d[1]);
                            d[2] = fmaf(w, v.z - me.z, d[2]);
                        }
                    }
                    d[0] += me.x;
                    d[1] += me.y;
                    d[2] += me.z;
                } else {
                    int ids[9];
                    lag_block(S, p, ids);
                    float lx[3], ly[3];
                    lag3(L.t[k - 1] * r * ex_of(k) - cx, lx[0], lx[1], lx[2]);
                    lag3(L.t[k - 1] * r * ey_of(k) - cy, ly[0], ly[1], ly[2]);
                    d[0] = d[1] = d[2] = 0.f;
                    for (int b = 0; b < 3; ++b)
                        for (int aa = 0; aa < 3; ++aa) {
                            const float w = lx[aa] * ly[b];
                            const float4 v = ruv[ids[b * 3 + aa]];
                            d[0] = fmaf(w, v.x, d[0]);
                            d[1] = fmaf(w, v.y, d[1]);
                            d[2] = fmaf(w, v.z, d[2]);
                        }
                }
                const float rd = 1.0f + d[0];
                val = geq(kp, d[0], rd, d[1], d[2]) + 0.5f * src(kp, rd, d[1], d[2], Cn.ax, Cn.ay);
            }
            fx += 2.0 * (double)val * ex_of(kp) * a;
            fy += 2.0 * (double)val * ey_of(kp) * a;
        }
    }
    // fixed-order block reduction
    __shared__ double sx[128], sy[128];
    sx[threadIdx.x] = fx;
    sy[threadIdx.x] = fy;
    __syncthreads();
    for (int h = 64; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) {
            sx[threadIdx.x] += sx[threadIdx.x + h];
            sy[threadIdx.x] += sy[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = sx[0];
        partial[2 * blockIdx.x + 1] = sy[0];
    }
}

// fixed-order sums of nb partial W-tuples (one block of 256)
template <int W>
__device__ __forceinline__ void sum_tuples(int nb, const double* __restrict__ partial, double* __restrict__ out) {
    double s[W];
#pragma unroll
    for (int q = 0; q < W; ++q) s[q] = 0.0;
    for (int b = threadIdx.x; b < nb; b += 256)
#pragma unroll
        for (int q = 0; q < W; ++q) s[q] += partial[W * (size_t)b + q];
    __shared__ double sh[W][256];
#pragma unroll
    for (int q = 0; q < W; ++q) sh[q][threadIdx.x] = s[q];
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h)
#pragma unroll
            for (int q = 0; q < W; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x < W) out[threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void __launch_bounds__(256) sum_pairs(int nb, const double* __restrict__ partial,
                                                 double* __restrict__ out) {
    sum_tuples<2>(nb, partial, out);
}

// ------------------------------------------------------------ reductions
// Six area-weighted FP64 sums: A, rho A, ux A, uy A, |u| A, |u|^2 A.
constexpr int kRedThreads = 256;

// the block's sums of s[W] into out[W], in a fixed order
template <int W>
__device__ __forceinline__ void block_tuple(const double* s, double* __restrict__ out) {
    __shared__ double sh[W][kRedThreads];
#pragma unroll
    for (int q = 0; q < W; ++q) sh[q][threadIdx.x] = s[q];
    __syncthreads();
    for (int h = kRedThreads / 2; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h)
#pragma unroll
            for (int q = 0; q < W; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x < W) out[threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void __launch_bounds__(kRedThreads, 4) reduce_fields_partial(int64_t n, const float* __restrict__ rho,
                                                                      const float* __restrict__ ux,
                                                                      const float* __restrict__ uy,
                                                                      const float* __restrict__ area,
                                                                      const uint8_t* __restrict__ mask,
                                                                      double* __restrict__ partial) {
    FieldSums t;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    // four nodes' loads in flight; the sums go on in node order
    for (; i + 3 * stride < n; i += 4 * stride) {
        float r[4], u[4], v[4], a[4];
        uint8_t m[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t k = i + j * stride;
            m[j] = mask ? mask[k] : 1;
            r[j] = rho[k];
            u[j] = ux[k];
            v[j] = uy[k];
            a[j] = area[k];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (m[j]) t.add(r[j], u[j], v[j], a[j]);
    }
    const bool few = n <= FieldSums::kFew * stride;
    for (; i < n; i += stride)
        if (!mask || mask[i]) {
            if (few) t.add64(rho[i], ux[i], uy[i], area[i]);
            else t.add(rho[i], ux[i], uy[i], area[i]);
        }
    t.flush();
    block_tuple<6>(t.s, partial + 6 * (size_t)blockIdx.x);
}

__global__ void __launch_bounds__(kRedThreads) reduce_fields_final(int nb, const double* __restrict__ partial,
                                                                    double* __restrict__ out) {
    sum_tuples<6>(nb, partial, out);
}

// Observables of every sample of a context in one launch, straight from the
// state (blockIdx.y is the sample; each has the block count it would have on
// its own, so its sums do not depend on the batch).
//   CHANGE: over masked nodes sum |u - u_prev|^2, sum |u|^2 and the number of
//   nodes whose density is not positive or whose fields are not finite, then
//   u into u_prev;  FIELDS: the six sums above.
// Partials [sample][max_nb][W], W = 3 or 6 (CHANGE first when both, W = 9).
__device__ __forceinline__ int blocks_of(int64_t m) {
    const int64_t b = (m + 4 * kRedThreads - 1) / (4 * kRedThreads);
    return (int)(b < 1 ? 1 : (b > kReduceMaxBlocks ? kReduceMaxBlocks : b));
}
template <int MODEL, bool CHANGE, bool FIELDS>
__global__ void __launch_bounds__(kRedThreads) observe_partial(const int64_t* __restrict__ seg, int max_nb,
                                                                const float4* __restrict__ st,
                                                                const float* __restrict__ f0, float ax0, float ay0,
                                                                const Collide* __restrict__ coll,
                                                                const float* __restrict__ area,
                                                                const uint8_t* __restrict__ mask,
                                                                float* __restrict__ px, float* __restrict__ py,
                                                                double* __restrict__ partial) {
    constexpr int W = (CHANGE ? 3 : 0) + (FIELDS ? 6 : 0);
    const int smp = blockIdx.y;
    const int64_t first = seg[smp], end = seg[smp + 1];
    const int nb = blocks_of(end - first);
    if ((int)blockIdx.x >= nb) return;
    const float ax = coll ? coll[smp].ax : ax0, ay = coll ? coll[smp].ay : ay0;
    double s[W];
#pragma unroll
    for (int q = 0; q < W; ++q) s[q] = 0.0;
    FieldSums t;
    const bool few = end - first <= FieldSums::kFew * (int64_t)nb * kRedThreads;
    for (int64_t i = first + blockIdx.x * (int64_t)kRedThreads + threadIdx.x; i < end; i += (int64_t)nb * kRedThreads) {
        float rho, u, v;
        if (MODEL == 0) {
            float dr;
            bgk_moments(st[2 * i], st[2 * i + 1], f0[i], ax, ay, dr, u, v);
            rho = 1.0f + dr;
        } else {
            const float4 a = st[i];
            rho = 1.0f + a.x;
            u = a.y;
            v = a.z;
        }
        if (mask[i]) {
            if (CHANGE) {
                if (!(rho > 0.f) || !isfinite(rho) || !isfinite(u) || !isfinite(v)) s[2] += 1.0;
                const double du = (double)u - px[i], dv = (double)v - py[i];
                s[0] += du * du + dv * dv;
                s[1] += (double)u * u + (double)v * v;
            }
            if (FIELDS) {
                if (few) t.add64(rho, u, v, area[i]);
                else t.add(rho, u, v, area[i]);
            }
        }
        if (CHANGE) {
            px[i] = u;
            py[i] = v;
        }
    }
    if (FIELDS) {
        t.flush();
#pragma unroll
        for (int q = 0; q < 6; ++q) s[(CHANGE ? 3 : 0) + q] = t.s[q];
    }
    block_tuple<W>(s, partial + W * ((size_t)smp * max_nb + blockIdx.x));
}

template <int W>
__global__ void __launch_bounds__(256) observe_final(const int64_t* __restrict__ seg, int max_nb,
                                                     const double* __restrict__ partial, double* __restrict__ out) {
    const int smp = blockIdx.x;
    sum_tuples<W>(blocks_of(seg[smp + 1] - seg[smp]), partial + W * ((size_t)smp * max_nb), out + W * (size_t)smp);
}

}  // namespace dev

cudaError_t launch_set_bgk(int n, const int* perm, const double* f, float4* f8, float* f0, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    dev::set_bgk_from_f64<<<blocks_for(n, 256), 256, 0, st>>>(n, perm, f, f8, f0);
    return cudaGetLastError();
}
cudaError_t launch_get_bgk(int n, const int* perm, const float4* f8, const float* f0, double* f, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    dev::get_bgk_to_f64<<<blocks_for(n, 256), 256, 0, st>>>(n, perm, f8, f0, f);
    return cudaGetLastError();
}
cudaError_t launch_set_bgk_equilibrium(int n, const int* perm, const double* ru, float4* f8, float* f0,
                                       cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    dev::set_bgk_equilibrium<<<blocks_for(n, 256), 256, 0, st>>>(n, perm, ru, f8, f0);
    return cudaGetLastError();
}
cudaError_t launch_set_tau1(int n, const int* perm, const double* ru, float4* s, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    dev::set_tau1_from_f64<<<blocks_for(n, 256), 256, 0, st>>>(n, perm, ru, s);
    return cudaGetLastError();
}
cudaError_t launch_macroscopics(int model, int n, const int* perm, const float4* f8, const float* f0,
                                const float4* ruv, float ax, float ay, const uint16_t* node_sample,
                                const dev::Collide* coll, int split, double* out, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    if (model == 0)
        dev::macroscopics_bgk<<<blocks_for(n, 256), 256, 0, st>>>(n, perm, f8, f0, ax, ay, node_sample, coll, split,
                                                                   out);
    else
        dev::macroscopics_tau1<<<blocks_for(n, 256), 256, 0, st>>>(n, perm, ruv, split, out);
    return cudaGetLastError();
}

int force_blocks(int n_link_nodes) { return std::max(1, std::min(256, blocks_for(n_link_nodes, 128))); }

cudaError_t launch_force(const dev::Stencil& S, int model, int n_link_nodes, const int* link_nodes,
                         const float* area_over_s2, const float4* f8, const float4* ruv, const dev::Collide& C,
                         double* partial, double* out, cudaStream_t st) {
    const int nb = force_blocks(n_link_nodes);
    if (S.Kq > 8) {
        MLBM_DISPATCH_KQ_RBF(S.Kq, (dev::force_kernel<KQC><<<nb, 128, 0, st>>>(S, model, n_link_nodes, link_nodes, area_over_s2, f8, ruv, C, partial)));
    } else {
        MLBM_DISPATCH_KQ(S.Kq, (dev::force_kernel<KQC><<<nb, 128, 0, st>>>(S, model, n_link_nodes, link_nodes, area_over_s2, f8, ruv, C, partial)));
    }
    dev::sum_pairs<<<1, 256, 0, st>>>(nb, partial, out);
    return cudaGetLastError();
}

int reduce_blocks(int64_t n) {
    const int64_t b = (n + 4 * dev::kRedThreads - 1) / (4 * dev::kRedThreads);
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, kReduceMaxBlocks));
}

cudaError_t launch_reduce_fields(const float* rho, const float* ux, const float* uy, const float* area,
                                 const uint8_t* mask, int64_t n, double* partial, double* out, cudaStream_t st) {
    // no more blocks than are resident at once: a second, partial round of them
    // would cost as much as the first
    const int nb = std::min(reduce_blocks(n), 4 * 152);
    dev::reduce_fields_partial<<<nb, dev::kRedThreads, 0, st>>>(n, rho, ux, uy, area, mask, partial);
    dev::reduce_fields_final<<<1, dev::kRedThreads, 0, st>>>(nb, partial, out);
    return cudaGetLastError();
}

cudaError_t launch_observe(int model, int what, int ns, int max_nb, const int64_t* seg, const float4* f8,
                           const float* f0, const float4* ruv, const dev::Collide& C, const dev::Collide* coll,
                           const float* area, const uint8_t* mask, float* px, float* py, double* partial, double* out,
                           cudaStream_t st) {
    const dim3 grid(max_nb, ns);
    auto run = [&](auto first, auto last) {
        first<<<grid, dev::kRedThreads, 0, st>>>(seg, max_nb, model == 0 ? f8 : ruv, f0, C.ax, C.ay, coll, area, mask,
                                                 px, py, partial);
        last<<<ns, 256, 0, st>>>(seg, max_nb, partial, out);
    };
    if (what == kObserveChange)
        model == 0 ? run(dev::observe_partial<0, true, false>, dev::observe_final<3>)
                   : run(dev::observe_partial<1, true, false>, dev::observe_final<3>);
    else if (what == kObserveFields)
        model == 0 ? run(dev::observe_partial<0, false, true>, dev::observe_final<6>)
                   : run(dev::observe_partial<1, false, true>, dev::observe_final<6>);
    else
        model == 0 ? run(dev::observe_partial<0, true, true>, dev::observe_final<9>)
                   : run(dev::observe_partial<1, true, true>, dev::observe_final<9>);
    return cudaGetLastError();
}

}  // namespace mlbm
