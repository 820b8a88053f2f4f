// Many BGK/TRT steps of a small set in one launch (variant 27): one cluster of
// blocks keeps the tile records and both state buffers in its shared memory.
//
// What bounds a step of a few thousand nodes is a chain of latencies: the
// launch, the gathers from L2 (~0.4 us), the stores' way back, the end of the
// grid.  Here block r of a cluster of up to 16 holds the tiles r * per .. of
// the set for a whole run, one a warp; members are read from the
// shared memory of the block that owns them, and the blocks meet at the
// cluster's hardware barrier after each step.  Global memory is read once
// before the first step and written once after the last.  The words that name
// a stencil's members in the records become their shared-memory addresses when
// the records have arrived.
#include <algorithm>

#include "device_common.cuh"
#include "kernels.h"
#include "launch_util.cuh"
#include "ring.cuh"
#include "step_node.cuh"

namespace mlbm {
namespace dev {

// all blocks of the cluster (one whose records never came steps nothing, but
// takes part in every barrier)
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of `at` in the shared memory of block `rank`
__device__ __forceinline__ uint32_t in_block(uint32_t at, uint32_t rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(at), "r"(rank));
    return a;
}
__device__ __forceinline__ float4 ld_cluster(uint32_t a) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float ld_cluster1(uint32_t a) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}

// States in the cluster's shared memory: member words are addresses in buffer
// 0, `buffer` bytes lead to the buffer that is read.
struct ClusterState {
    uint32_t buffer;
    const float4* own;     // the lane's own state in that buffer
    const LinkRec* links;  // the lane's links, where it has any
    __device__ __forceinline__ void pair(int j, float4& a, float4& b) const {
        a = ld_cluster((uint32_t)j + buffer);
        b = ld_cluster((uint32_t)j + buffer + 16);
    }
    __device__ __forceinline__ float at(int j, int k) const { return ld_cluster1((uint32_t)j + buffer + 4 * (k - 1)); }
};

// Increments of the eight streamed populations over the node's own.  AHEAD
// groups of gathers are in flight; those of group q + AHEAD go out member by
// member as group q is used up.
// LINK: a direction that is a link takes the reflected population at its own
// point x + t s e_k (t = tt[k-1] = 1 - 2q), from the same rows: with x = t e
// the weight is m0 (1 - t^2) + t^2 U +- t m1 (and V, W, W' in turn).
template <int KQ, bool LINK, int AHEAD>
__device__ __forceinline__ void wls_increments(const ClusterState& st, const float4* base, const int4* id,
                                               const float4& oa, const float4& ob, uint32_t mask, const float* tt,
                                               float* acc) {
    constexpr int kSp = TileRec<KQ>::kSp;
    float4 fa[4 * AHEAD], fb[4 * AHEAD];
#pragma unroll
    for (int j = 0; j < 4 * AHEAD; ++j)
        if (j != 4 * kSp + 3) st.pair(at4(id[j / 4], j % 4), fa[j], fb[j]);
#pragma unroll
    for (int q = 0; q < KQ; ++q) {
        float4 m[6];
        slot_rows<KQ>(base, q, m);
        float4* ga = fa + 4 * (q % AHEAD);
        float4* gb = fb + 4 * (q % AHEAD);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (q != kSp || c != 3) {
                const float d[8] = {ga[c].x - oa.x, ga[c].y - oa.y, ga[c].z - oa.z, ga[c].w - oa.w,
                                    gb[c].x - ob.x, gb[c].y - ob.y, gb[c].z - ob.z, gb[c].w - ob.w};
                const float U = at4(m[0], c), V = at4(m[1], c), Wd = at4(m[2], c), Wp = at4(m[3], c),
                            m1 = at4(m[4], c), m2 = at4(m[5], c);
                if (!LINK) {
                    wls_acc_diff(d[0], d[1], d[2], d[3], d[4], d[5], d[6], d[7], U, V, Wd, Wp, m1, m2, acc);
                } else {
                    const float m0 = (U + V) - 0.5f * (Wd + Wp);
                    const float quad[8] = {U, V, U, V, Wd, Wp, Wd, Wp};
                    const float gs = m1 + m2, hs = m1 - m2;
                    const float lin[8] = {m1, m2, -m1, -m2, gs, -hs, -gs, hs};
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float t2 = tt[k] * tt[k];
                        const float a = ((mask >> (k + 1)) & 1u) ? d[opp_of(k + 1) - 1] : d[k];
                        acc[k] = fmaf(tt[k] * lin[k], a, fmaf(fmaf(1.f - t2, m0, t2 * quad[k]), a, acc[k]));
                    }
                }
            }
            if (q + AHEAD < KQ && !(q + AHEAD == kSp && c == 3))
                st.pair(at4(id[(q + AHEAD) % KQ], c), ga[c], gb[c]);
        }
    }
}

// One step of node p, whose lane of the record is `base` and whose index rows
// are in id: (o0, o1, rest).  The same arithmetic as a launch per step
// (walk_tiles), bit for bit.
template <int KQ, int AHEAD>
__device__ __forceinline__ void cluster_node(const Stencil& S, const ClusterState& st, const Collide& C,
                                             const float4* base, const int4* id, int p, float4& o0, float4& o1,
                                             float& rest) {
    using R = TileRec<KQ>;
    const int word = id[R::kSp].w;
    const uint8_t meta = (uint8_t)(word & 0xff);
    const int kind = meta & 3;
    float4 oa = make_float4(0, 0, 0, 0), ob = oa;
    float f0own = 0.f;
    float acc[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = 0.f;
    LinkRec lk;
    lk.mask = 0;
    const bool links = (meta & 4) && kind != 2;
    if (kind != 2) {
        oa = st.own[0];
        ob = st.own[1];
        f0own = rest;
    }
    if (links) lk = *st.links;
    const bool moved = S.bb_mode != 0 && __any_sync(0xffffffffu, links && kind == 0);
    if (kind == 0) {
        if (moved) {
            float tt[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) tt[k] = ((lk.mask >> (k + 1)) & 1u) ? lk.t[k] : -1.0f;
            wls_increments<KQ, true, AHEAD>(st, base, id, oa, ob, lk.mask, tt, acc);
        } else {
            wls_increments<KQ, false, AHEAD>(st, base, id, oa, ob, 0u, nullptr, acc);
        }
    }
    float g[9];
    if (kind == 2) {
        const float4 e = S.eqv[p];
        eq_populations(e.x, e.y, e.z, g);
    } else {
        const float own[8] = {oa.x, oa.y, oa.z, oa.w, ob.x, ob.y, ob.z, ob.w};
        if (kind == 0) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const bool lnk = (lk.mask >> (k + 1)) & 1u;
                const float o = lnk ? own[opp_of(k + 1) - 1] : own[k];
                g[k + 1] = lnk && S.bb_mode == 0 ? o : acc[k] + o;
            }
        } else if constexpr (KQ >= 3) {
            const int ids[9] = {id[0].x, id[0].y, id[0].z, id[0].w, id[1].x, id[1].y, id[1].z, id[1].w, id[2].x};
            const float r = __int_as_float(id[2].y), cx = (float)ex_of(meta >> 4), cy = (float)ey_of(meta >> 4);
            lagrange_increments<1>([&](int j, float4& a, float4& b) { st.pair(j, a, b); }, ids, r, cx, cy, oa, ob,
                                   0, acc);
#pragma unroll
            for (int k = 0; k < 8; ++k) g[k + 1] = acc[k] + own[k];
            if (links)
#pragma unroll
                for (int k = 1; k < 9; ++k) {
                    if (!((lk.mask >> k) & 1u)) continue;
                    const int kp = opp_of(k);
                    g[k] = S.bb_mode == 0 ? own[kp - 1]
                                          : lagrange_link([&](int j, int kk) { return st.at(j, kk); }, ids, r, cx,
                                                          cy, k, lk.t[k - 1], own[kp - 1]);
                }
        }
        g[0] = f0own;
        collide_pairs(g, C, 0xFu, true);
    }
    o0 = make_float4(g[1], g[2], g[3], g[4]);
    o1 = make_float4(g[5], g[6], g[7], g[8]);
    rest = g[0];
}

// Tiles (and warps) of a block.  More of them share the block's and the cluster's
// shared-memory ports, and at eight launches of dependent grids are as fast, or
// faster from K = 16 on (K = 12 is still 7% ahead there; one limit serves every
// K).  us a step, launches / cluster, at 500 nodes (one tile a block), 2000
// (four) and 3774 (eight): K = 12 2.97 / 1.85, 2.97 / 1.98, 3.10 / 2.90; K = 16
// 3.22 / 2.26, 3.27 / 2.71, 3.48 / 3.83; K = 24 4.14 / 3.54, 4.43 / 3.93, 4.60 /
// 5.56.  (With the states in L2 and the same barrier: 2.18 at 2000 nodes, K = 12.)
constexpr int kClusterWarps = 4;

template <int KQ>
__global__ void __launch_bounds__(kClusterWarps * 32, 1)
    step_cluster(Stencil S, const float4* in, const float* f0in, float4* out, float* f0out, Collide C0, int per,
                 int steps, int* err, const Wait W) {
    constexpr int kBytes = TileRec<KQ>::kRows * 512;
    constexpr int kState = 2;  // float4 of a node's moving populations
    constexpr int kAhead = KQ <= 4 ? KQ : (KQ == 6 ? 3 : 2);  // groups of gathers in flight: all that 255 registers hold
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t bar;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles = (S.n + 31) / 32, t0 = blockIdx.x * per, nt = max(0, min(per, tiles - t0));
    // states behind the records: buffer b of tile i at (b * per + i) * 32 nodes
    float4* states = reinterpret_cast<float4*>(smem + (size_t)per * kBytes);
    const uint32_t buffer_bytes = (uint32_t)per * 32 * kState * 16;
    const bool withhold = W.withhold && blockIdx.x == 0;  // test switch: the block's copies are never issued
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (threadIdx.x == 0 && !withhold) {  // what each tile needs of its record (see step_warp), all on one barrier
        uint32_t bytes = 0;
        for (int i = 0; i < nt; ++i) {
            const int need = S.need[t0 + i];
            bytes += need == 2 ? kBytes : (need == 1 ? 3 * 512 : 512);
        }
        mbar_expect_tx(&bar, bytes);
        for (int i = 0; i < nt; ++i) {
            const int need = S.need[t0 + i];
            const int first = need == 0 ? TileRec<KQ>::kSp * 512 : 0;
            bulk_g2s(smem + (size_t)i * kBytes + first,
                     reinterpret_cast<const uint8_t*>(S.rec) + (size_t)(t0 + i) * kBytes + first,
                     need == 2 ? kBytes : (need == 1 ? 3 * 512 : 512), &bar);
        }
    }
    // the lane's node: its state, and later its rest population, in registers
    const int p = (t0 + warp) * 32 + lane;
    const bool live = warp < nt && p < S.n;
    float4* own = states + (size_t)(warp * 32 + lane) * kState;  // in buffer 0
    const size_t other = (size_t)per * 32 * kState;
    LinkRec* links = reinterpret_cast<LinkRec*>(states + 2 * other) + warp * 32 + lane;
    float rest = 0.f;
    if (live) {
        own[0] = in[(size_t)p * kState];
        own[1] = in[(size_t)p * kState + 1];
        rest = f0in[p];
        if (S.meta[p] & 4) *links = S.links[S.link_slot[p]];
    }
    __syncthreads();
    // a block whose records never came steps nothing, but stays: the others read its states
    const bool ok = __syncthreads_and(mbar_wait(&bar, 0, W.budget_ns));
    if (!ok && threadIdx.x == 0) {
        atomicExch(err, 2);
        if (!withhold) mbar_wait(&bar, 0, W.budget_ns);  // do not leave while copies may still be landing
    }
    const float4* base = reinterpret_cast<const float4*>(smem + (size_t)warp * kBytes) + lane;
    const bool mine = ok && warp < nt;
    int4 id[KQ];
    Collide C = C0;
    if (mine) {
#pragma unroll
        for (int q = 0; q < KQ; ++q) id[q] = reinterpret_cast<const int4*>(base)[q * 32];
        if (S.coll) C = S.coll[id[TileRec<KQ>::kSp].w >> 8];
        // positions of members -> their addresses
        const int kind = id[TileRec<KQ>::kSp].w & 3, members = kind == 0 ? 4 * KQ : (kind == 1 ? 9 : 0);
        const uint32_t first = saddr(states);
        auto address = [&](int j, int& word) {
            if (j >= members || j == 4 * TileRec<KQ>::kSp + 3) return;
            const int t = word >> 5, rank = t / per;
            word = (int)in_block(first + (uint32_t)((t - rank * per) * 32 + (word & 31)) * (kState * 16), rank);
        };
#pragma unroll
        for (int q = 0; q < KQ; ++q) {
            address(4 * q, id[q].x);
            address(4 * q + 1, id[q].y);
            address(4 * q + 2, id[q].z);
            address(4 * q + 3, id[q].w);
        }
    }
    cluster_barrier();  // every block's states are there
    float4 o0 = make_float4(0.f, 0.f, 0.f, 0.f), o1 = o0;
    for (int s = 0; s < steps; ++s) {
        const bool odd = s & 1;
        if (mine) {
            const ClusterState st{odd ? buffer_bytes : 0u, odd ? own + other : own, links};
            // Nothing is to be computed once for all steps: a product taken out of
            // the loop would be rounded apart from the sum that it is fused with
            // in a kernel of one step, and the states would differ.
            asm volatile("" : "+f"(C.omega_p), "+f"(C.omega_m), "+f"(C.src_p), "+f"(C.src_m), "+f"(C.ax), "+f"(C.ay));
#pragma unroll
            for (int q = 0; q < KQ; ++q) asm volatile("" : "+r"(id[q].x), "+r"(id[q].y), "+r"(id[q].z), "+r"(id[q].w));
            cluster_node<KQ, kAhead>(S, st, C, base, id, p, o0, o1, rest);
            float4* to = odd ? own : own + other;
            to[0] = o0;
            to[1] = o1;
        }
        cluster_barrier();  // after the last step too: others may still read this block's states
    }
    if (live && ok) {
        out[(size_t)p * kState] = o0;
        out[(size_t)p * kState + 1] = o1;
        f0out[p] = rest;
    }
}

}  // namespace dev

namespace {

constexpr int kMaxShared = 226 << 10;  // and 1 KB for the block's own

// shared memory of a tile: its record, two buffers of states, links
template <int KQ>
constexpr int tile_bytes() {
    return dev::TileRec<KQ>::kRows * 512 + 2 * 32 * 32 + 32 * (int)sizeof(dev::LinkRec);
}

// A launch of one cluster of `size` blocks
template <int KQ, class F>
cudaError_t with_cluster(int tiles, int size, cudaStream_t st, F go) {
    const int per = (tiles + size - 1) / size;
    const size_t tile = tile_bytes<KQ>();
    auto fn = dev::step_cluster<KQ>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxShared);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)size);
    cfg.blockDim = dim3((unsigned)(per * 32));
    cfg.dynamicSmemBytes = per * tile;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)size;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return go(fn, cfg, per);
}

template <int KQ>
int cluster_for(int n) {
    const int tiles = (n + 31) / 32;
    for (int size = 16; size >= 1; size /= 2) {
        if (size > tiles) continue;
        const int per = (tiles + size - 1) / size;
        if (per > dev::kClusterWarps || per * tile_bytes<KQ>() > kMaxShared) return 0;
        int clusters = 0;
        const cudaError_t e = with_cluster<KQ>(tiles, size, nullptr, [&](auto fn, const cudaLaunchConfig_t& cfg, int) {
            return cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg);
        });
        if (e == cudaSuccess && clusters > 0) return size;
        (void)cudaGetLastError();  // the device takes no cluster of this size
    }
    return 0;
}

}  // namespace

int step_cluster_size(int Kq, int n) {
    if (n < 1) return 0;
    switch (Kq) {
        case 3: return cluster_for<3>(n);
        case 4: return cluster_for<4>(n);
        case 6: return cluster_for<6>(n);
        case 8: return cluster_for<8>(n);
        default: return 0;
    }
}

namespace {
template <int KQ>
cudaError_t run_cluster(int size, const dev::Stencil& S, const float4* in, const float* f0in, float4* out,
                        float* f0out, const dev::Collide& C, int steps, int* err, const dev::Wait& W,
                        cudaStream_t st) {
    return with_cluster<KQ>((S.n + 31) / 32, size, st, [&](auto fn, const cudaLaunchConfig_t& cfg, int per) {
        return cudaLaunchKernelEx(&cfg, fn, S, in, f0in, out, f0out, C, per, steps, err, W);
    });
}
}  // namespace

cudaError_t launch_step_cluster(int size, const dev::Stencil& S, const float4* in, const float* f0in, float4* out,
                                float* f0out, const dev::Collide& C, int steps, int* err, const dev::Wait& W,
                                cudaStream_t st) {
    switch (S.Kq) {
        case 3: return run_cluster<3>(size, S, in, f0in, out, f0out, C, steps, err, W, st);
        case 4: return run_cluster<4>(size, S, in, f0in, out, f0out, C, steps, err, W, st);
        case 6: return run_cluster<6>(size, S, in, f0in, out, f0out, C, steps, err, W, st);
        case 8: return run_cluster<8>(size, S, in, f0in, out, f0out, C, steps, err, W, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace mlbm
