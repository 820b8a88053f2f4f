// BGK/TRT step on RBF-FD stencils from tile records that hold the non-zero
// weights only, streamed by independent warps.
//
// What bounds the step is the weight rows: a stencil per Lagrangian point
// (25 nodes each, a union of up to 64 slots) stores 8 x 64 weights and 64
// positions a node, 2.3 KB of which only 8 x 25 weights are not zero; 65k
// nodes read 150 MB a step from HBM.  A record keeps, for half the directions
// of 16 nodes (lane 2 i + h: directions 4 h + 1 .. 4 h + 4 of node i),
//   groups x 512 B   the members of the half's stencils, four int4 words a
//                    lane: position, and in the top four bits the directions
//                    that have a weight for it
//   rows x 128 B     the lane's weights in the order they are used
// (1.1 KB a node, 71 MB, which stays in L2).  A lane reads the weight at its
// own place in its own column, so whatever the places of a warp's lanes, the
// reads meet no bank conflict; a gather is the 16 bytes that the half needs.
// The weights that are left out add zero, and the others are added in the
// slot order of the plain kernel: the same state bit for bit.
// One warp owns one shared-memory slot, which a bulk copy refills while the
// warp collides and stores; what bounds it now is the chain of a tile, a dozen
// rounds of gathers and weight reads, on the ten warps whose slots an SM holds
// (34% of issue slots, stalls on gathers and records).
// us a step, plain rows / records: 65k nodes 25.4 / 18.8, 46k 20.9 / 13.5.  (A
// branch for each weight 24.3, three groups of gathers ahead with spills 22.0.)
#include <algorithm>
#include <vector>

#include "device_common.cuh"
#include "kernels.h"
#include "launch_util.cuh"
#include "ring.cuh"
#include "step_node.cuh"

namespace mlbm {
namespace dev {

constexpr int kHalfNodes = 16;  // nodes of a tile

// which of the half's four weights of slots 4 q .. 4 q + 3 are not zero: bit
// 4 c + b for slot c, direction 4 h + 1 + b
__device__ __forceinline__ unsigned half_bits(const Stencil& S, int p, int h, int q, float w[4][4]) {
    unsigned bits = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const float4 v = S.Wr[(size_t)((4 * h + b) * S.Kq + q) * S.n_pad + p];
        w[b][0] = v.x; w[b][1] = v.y; w[b][2] = v.z; w[b][3] = v.w;
#pragma unroll
        for (int c = 0; c < 4; ++c) bits |= (w[b][c] != 0.f ? 1u : 0u) << (4 * c + b);
    }
    return bits;
}

// (member groups, weight rows) of every tile
__global__ void __launch_bounds__(128) rbf_tile_sizes(Stencil S, int tiles, int2* __restrict__ size) {
    const int tile = (int)((blockIdx.x * 128LL + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (tile >= tiles) return;
    const int p = tile * kHalfNodes + (lane >> 1), h = lane & 1;
    int members = 0, weights = 0;
    if (p < S.n) {
        const int kind = S.meta[p] & 3;
        if (kind == 1) members = 9;
        for (int q = 0; kind == 0 && q < S.Kq; ++q) {
            float w[4][4];
            const unsigned bits = half_bits(S, p, h, q, w);
            weights += __popc(bits);
#pragma unroll
            for (int c = 0; c < 4; ++c) members += ((bits >> (4 * c)) & 15u) != 0;
        }
    }
    members = __reduce_max_sync(0xffffffffu, members);
    weights = __reduce_max_sync(0xffffffffu, weights);
    if (lane == 0) size[tile] = make_int2((members + 3) / 4, weights);
}

__global__ void __launch_bounds__(128) rbf_tile_fill(Stencil S, int tiles, const int4* __restrict__ head,
                                                     uint8_t* __restrict__ rec) {
    const int tile = (int)((blockIdx.x * 128LL + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (tile >= tiles) return;
    const int p = tile * kHalfNodes + (lane >> 1), h = lane & 1;
    const int4 hd = head[tile];
    int* id = reinterpret_cast<int*>(rec + (size_t)hd.x * 128) + lane * 4;            // member m: id[(m / 4) * 128 + m % 4]
    float* wt = reinterpret_cast<float*>(rec + (size_t)hd.x * 128 + hd.y * 512) + lane;  // weight r: wt[r * 32]
    int m = 0, r = 0;
    auto put = [&](int j, unsigned mask) {
        id[(m >> 2) * 128 + (m & 3)] = j | (int)(mask << 28);
        ++m;
    };
    if (p < S.n) {
        const int kind = S.meta[p] & 3;
        if (kind == 1) {
            int ids[9];
            lag_block(S, p, ids);
            for (int b = 0; b < 9; ++b) put(ids[b], 0u);
        }
        for (int q = 0; kind == 0 && q < S.Kq; ++q) {
            float w[4][4];
            const unsigned bits = half_bits(S, p, h, q, w);
            const int4 i4 = S.idx[(size_t)q * S.n_pad + p];
            const int ids[4] = {i4.x, i4.y, i4.z, i4.w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const unsigned mask = (bits >> (4 * c)) & 15u;
                if (!mask) continue;
                put(ids[c], mask);
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if ((mask >> b) & 1u) wt[32 * r++] = w[b][c];
            }
        }
    }
    while (m < 4 * hd.y) put(p < S.n ? p : 0, 0u);
    for (; r < hd.z; ++r) wt[32 * r] = 0.f;
}

// The half's increments over the node's own populations, from the warp's slot.
// LINK: a direction whose bit is set in `links` takes the opposite population
// (of the same half) at its own point, the reflected one.
template <bool LINK>
__device__ __forceinline__ void half_increments(const float4* __restrict__ f, const int4* ids, const float* wt,
                                                int groups, int h, const float4& own, unsigned links, float* acc) {
    if (groups == 0) return;  // every direction of the tile's nodes is a simple bounce-back link
    auto at = [&](int word) { return __ldg(f + 2 * (size_t)(word & 0x0fffffff) + h); };
    // a lane's next weight; beyond its last one, at most one row, lies slot too
    const char* next = reinterpret_cast<const char*>(wt);
    auto use = [&](const int4& id, const float4* v) {
        const int word[4] = {id.x, id.y, id.z, id.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float d[4] = {v[c].x - own.x, v[c].y - own.y, v[c].z - own.z, v[c].w - own.w};
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                // no branch: a weight that another direction or member owns is read and dropped
                const float w = *reinterpret_cast<const float*>(next);
                const int step = (int)((unsigned)word[c] >> (21 + b)) & 128;
                const float x = LINK && ((links >> b) & 1u) ? d[b ^ 2] : d[b];
                const float sum = fmaf(w, x, acc[b]);
                acc[b] = step ? sum : acc[b];
                next += step;
            }
        }
    };
    // two groups of four gathers in flight while a third is used
    int4 ia = ids[0], ib = groups > 1 ? ids[32] : ia;
    float4 a[4] = {at(ia.x), at(ia.y), at(ia.z), at(ia.w)}, b[4] = {at(ib.x), at(ib.y), at(ib.z), at(ib.w)};
    for (int g = 0; g < groups; g += 2) {
        use(ia, a);
        if (g + 2 < groups) {
            ia = ids[(g + 2) * 32];
            a[0] = at(ia.x);
            a[1] = at(ia.y);
            a[2] = at(ia.z);
            a[3] = at(ia.w);
        }
        if (g + 1 < groups) use(ib, b);
        if (g + 3 < groups) {
            ib = ids[(g + 3) * 32];
            b[0] = at(ib.x);
            b[1] = at(ib.y);
            b[2] = at(ib.z);
            b[3] = at(ib.w);
        }
    }
}

// this half's increments of a Lagrange node (the terms and order of lagrange_increments)
__device__ __forceinline__ void lagrange_half(const float4* __restrict__ f, const int* ids, float r, float cx, float cy,
                                              int h, const float4& own, float* acc) {
    float xp[3], x0[3], xm[3], yp[3], y0[3], ym[3];
    lag3(-r - cx, xp[0], xp[1], xp[2]);
    lag3(-cx, x0[0], x0[1], x0[2]);
    lag3(r - cx, xm[0], xm[1], xm[2]);
    lag3(-r - cy, yp[0], yp[1], yp[2]);
    lag3(-cy, y0[0], y0[1], y0[2]);
    lag3(r - cy, ym[0], ym[1], ym[2]);
#pragma unroll
    for (int bp = 0; bp < 9; ++bp) {
        const int b = bp / 3, a = bp % 3;
        const float4 v = __ldg(f + 2 * (size_t)ids[bp] + h);
        acc[0] = fmaf(h ? xp[a] * yp[b] : xp[a] * y0[b], v.x - own.x, acc[0]);
        acc[1] = fmaf(h ? xm[a] * yp[b] : x0[a] * yp[b], v.y - own.y, acc[1]);
        acc[2] = fmaf(h ? xm[a] * ym[b] : xm[a] * y0[b], v.z - own.z, acc[2]);
        acc[3] = fmaf(h ? xp[a] * ym[b] : x0[a] * ym[b], v.w - own.w, acc[3]);
    }
}

__global__ void __launch_bounds__(kRbfMaxWarps * 32, 1)
    step_rbf_tiles(Stencil S, const float4* __restrict__ in, const float* __restrict__ f0in, float4* __restrict__ out,
                   float* __restrict__ f0out, Collide C0, int backward, int* __restrict__ err, const Wait W) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int lane = threadIdx.x & 31;
    uint8_t* slot = smem + (size_t)warp * S.rbf_slot;
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + (size_t)warps * S.rbf_slot) + warp;
    const int t0 = S.rbf_range[blockIdx.x], t1 = S.rbf_range[blockIdx.x + 1];
    if (warp >= t1 - t0) return;
    int t = backward ? t1 - 1 - warp : t0 + warp;
    const int hop = backward ? -warps : warps;
    // lane 0: the slot's barrier completes when the tile's record is there (a
    // tile of equilibrium nodes has none)
    auto fetch = [&](const int4& hd) {
        const uint32_t bytes = (uint32_t)(hd.y * 512 + hd.z * 128);
        mbar_expect_tx(bar, bytes);
        if (bytes) bulk_g2s(slot, S.rbf_rec + (size_t)hd.x * 128, bytes, bar);
    };
    int4 head = S.rbf_head[t];
    if (lane == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        fetch(head);
    }
    __syncwarp();
    pdl_trigger();
    pdl_wait();
    const int h = lane & 1;
    uint32_t ph = 0;
    for (; t >= t0 && t < t1; t += hop) {
        const int tn = t + hop;
        const bool last = tn < t0 || tn >= t1;
        const int p = t * kHalfNodes + (lane >> 1);
        const bool live = p < S.n;
        const uint8_t meta = live ? S.meta[p] : (uint8_t)2;
        const int kind = meta & 3;
        const int4 next = last ? make_int4(0, 0, 0, 0) : S.rbf_head[tn];
        float4 own = make_float4(0.f, 0.f, 0.f, 0.f);
        float f0own = 0.f;
        unsigned links = 0;  // of the half's directions
        if (kind != 2) {
            own = __ldg(in + 2 * (size_t)p + h);
            f0own = f0in[p];
            if (meta & 4) links = (S.links[S.link_slot[p]].mask >> (4 * h + 1)) & 15u;
        }
        if (!__all_sync(0xffffffffu, mbar_wait(bar, ph, W.budget_ns))) {
            if (lane == 0) {
                atomicExch(err, 2);
                mbar_wait(bar, ph, W.budget_ns);  // do not leave while the record may still be landing
            }
            return;
        }
        ph ^= 1u;
        const int4* ids = reinterpret_cast<const int4*>(slot) + lane;
        const float* wt = reinterpret_cast<const float*>(slot + (size_t)head.y * 512) + lane;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        const bool moved = S.bb_mode != 0 && __any_sync(0xffffffffu, kind == 0 && links != 0);
        const float o[4] = {own.x, own.y, own.z, own.w};
        float s[4], x[4];
        if (kind == 0) {
            if (moved) half_increments<true>(in, ids, wt, head.y, h, own, links, acc);
            else half_increments<false>(in, ids, wt, head.y, h, own, 0u, acc);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const bool lnk = (links >> b) & 1u;
                s[b] = lnk && S.bb_mode == 0 ? o[b ^ 2] : acc[b] + (lnk ? o[b ^ 2] : o[b]);
            }
        } else if (kind == 1) {
            const int4 i0 = ids[0], i1 = ids[32], i2 = ids[64];
            const int block[9] = {i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, i1.z, i1.w, i2.x};
            const float r = S.lag_r[p], cx = (float)ex_of(meta >> 4), cy = (float)ey_of(meta >> 4);
            lagrange_half(in, block, r, cx, cy, h, own, acc);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                s[b] = acc[b] + o[b];
                if ((links >> b) & 1u)
                    s[b] = S.bb_mode == 0 ? o[b ^ 2]
                                          : lagrange_link([&](int j, int k) { return pop(in, j, k); }, block, r, cx, cy, 4 * h + 1 + b,
                                                          S.links[S.link_slot[p]].t[4 * h + b], o[b ^ 2]);
            }
        }
        __syncwarp();
        if (lane == 0 && !last) fetch(next);
        head = next;
#pragma unroll
        for (int b = 0; b < 4; ++b) x[b] = __shfl_xor_sync(0xffffffffu, s[b], 1);
        float g[9];
        if (kind == 2) {
            const float4 e = live ? S.eqv[p] : own;
            eq_populations(e.x, e.y, e.z, g);
        } else {
            g[0] = f0own;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                g[1 + b] = h ? x[b] : s[b];
                g[5 + b] = h ? s[b] : x[b];
            }
            collide_pairs(g, collide_of(S, C0, p), 0xFu, true);
        }
        if (live) {
            out[2 * (size_t)p + h] = h ? make_float4(g[5], g[6], g[7], g[8]) : make_float4(g[1], g[2], g[3], g[4]);
            if (h == 0) f0out[p] = g[0];
        }
    }
}

}  // namespace dev

namespace {
// shared memory of a block's slots: more warps are worth more here than the L1
// they leave to the gathers (65k nodes: 22.0 us with 168 KB, 20.2 with 216 KB)
constexpr int kRbfSlotBytes = 216 << 10;
// see kResident of the least-squares step: above this many bytes of records
// steps walk the tiles forwards and backwards in turn
constexpr size_t kRbfResident = size_t(100) << 20;

int rbf_warps(int slot) { return std::max(1, std::min(dev::kRbfMaxWarps, kRbfSlotBytes / (slot + 8))); }
}  // namespace

cudaError_t rbf_tile_sizes(const dev::Stencil& S, int tiles, int2* size, cudaStream_t st) {
    if (tiles == 0) return cudaSuccess;
    dev::rbf_tile_sizes<<<(tiles + 3) / 4, 128, 0, st>>>(S, tiles, size);
    return cudaGetLastError();
}

cudaError_t rbf_tile_fill(const dev::Stencil& S, int tiles, const int4* head, uint8_t* rec, cudaStream_t st) {
    if (tiles == 0) return cudaSuccess;
    dev::rbf_tile_fill<<<(tiles + 3) / 4, 128, 0, st>>>(S, tiles, head, rec);
    return cudaGetLastError();
}

bool rbf_tiles_plan(const std::vector<int2>& size, int blocks, std::vector<int4>& head, std::vector<int>& range,
                    int& slot, size_t& bytes) {
    const int tiles = (int)size.size();
    head.resize(size.size());
    size_t units = 0, widest = 0;  // of 128 bytes
    for (int t = 0; t < tiles; ++t) {
        head[(size_t)t] = make_int4((int)units, size[(size_t)t].x, size[(size_t)t].y, 0);
        const size_t u = 4 * (size_t)size[(size_t)t].x + (size_t)size[(size_t)t].y;
        units += u;
        widest = std::max(widest, u);
    }
    bytes = units * 128;
    slot = (int)((widest + 1) * 128);  // and the row a lane may read past its weights
    if (units > (size_t)1 << 30 || slot > 96 << 10) return false;
    // ranges of equal cost: the record's bytes, and the state each tile moves
    const size_t per_tile = 12, total = units + per_tile * (size_t)tiles;
    range.assign((size_t)blocks + 1, tiles);
    size_t before = 0;
    int b = 0;
    for (int t = 0; t < tiles; ++t) {
        for (; b < blocks && before * (size_t)blocks >= total * (size_t)b; ++b) range[(size_t)b] = t;
        before += per_tile + 4 * (size_t)size[(size_t)t].x + (size_t)size[(size_t)t].y;
    }
    return true;
}

cudaError_t launch_step_rbf_tiles(const dev::Stencil& S, const float4* in, const float* f0in, float4* out,
                                  float* f0out, const dev::Collide& C, int backward, int* err, const dev::Wait& W,
                                  cudaStream_t st) {
    if (S.n == 0) return cudaSuccess;
    const int warps = rbf_warps(S.rbf_slot);
    const size_t smem = (size_t)warps * (S.rbf_slot + 8);
    const cudaError_t e =
        cudaFuncSetAttribute(dev::step_rbf_tiles, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int back = S.rbf_bytes > kRbfResident ? backward : 0;
    return launch_pdl_smem(dev::step_rbf_tiles, S.rbf_blocks, warps * 32, smem, st, S, in, f0in, out, f0out, C, back,
                           err, W);
}

}  // namespace mlbm
