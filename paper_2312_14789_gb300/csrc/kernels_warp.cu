// Step kernels whose warps stream their own node tiles (variants 27-29), and
// the tile bookkeeping they need.
//
// What bounds a step is how many bytes of stencil rows an SM keeps in flight.
// A thread that loads its rows into registers holds about ten 16-byte loads at
// 128 registers and waits for them group by group: 16 warps an SM moved 5.8
// TB/s on a 192k-node tau = 1 sample whose rows sit in L2, and 0.85 of the
// copy rate on a 1.7M-node batch.  Here a warp owns one shared-memory slot,
// the record of one 32-node tile (13.8 KB at K = 16), and refills it with two
// bulk copies (index rows, matrix rows) the moment it has read them, so the
// next tile's rows fly while the warp collides, stores and waits for its own
// gathers, and no register holds a row.  No warp waits for another one.
//   - Twelve slots (166 KB) leave 62 KB of L1 to the gathers and 168 registers
//     a thread: enough for all 15 gathers of a tau = 1 node, or for a BGK
//     node's group of four with one register spilled (K = 32, eight slots: 16).
//     16 slots spill and starve the L1 (BGK vortex street, 260k nodes: 31 us
//     against 23 with 12).
//   - A block takes one contiguous range of tiles (neighbouring tiles share
//     gathers in L1); the ranges are cut to equal cost, because tiles of a
//     regular region fetch index rows only.
//   - With interpolated bounce-back a warp that has link nodes evaluates every
//     direction at its own point in the same pass (a lane without links uses
//     t = -1, which reproduces the plain weights bit for bit), where one thread
//     used to walk its stencil again for each link.
//   - When the records outgrow L2, steps walk the tiles forwards and backwards
//     in turn, so that a step starts on what the last one left in L2.
// Step times before (variant 25, rows loaded by each thread) and after, us,
// K = 16, graph replay on one GB300: 2k-node channel (K = 12) 5.2 / 2.9; 192k
// porous tau = 1 15.7 / 14.3; nine flows of it, 1.73M nodes, 142.4 / 120.1
// (6.7 TB/s of stored bytes); 96k porous TRT with interpolated links 24.5 /
// 8.1; vortex street 260k 25.3 / 20.4; its hybrid set, 165k, 13.1 / 9.8.
#include <algorithm>

#include "device_common.cuh"
#include "kernels.h"
#include "launch_util.cuh"
#include "ring.cuh"
#include "step_node.cuh"

namespace mlbm {
namespace dev {

// loads kept in program order, so that the gathers of a node go out together
__device__ __forceinline__ float4 ldg_now(const float4* p) {
    float4 v;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ void ldg_pair_now(const float4* p, float4& a, float4& b) {
    asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(p));
}

// relative time of a tile by what it fetches (the hybrid vortex street, whose
// tiles of all three sorts lie in separate regions, took 13.3 us with equal
// tile counts and 9.8 us with these)
constexpr int kCostCopy = 1, kCostLagrange = 2, kCostStencil = 5;

template <int KQ, int WARPS>
struct WarpTile {
    static constexpr int kBytes = TileRec<KQ>::kRows * 512;
    static constexpr int kWarps = WARPS;
    static constexpr int kSmem = kWarps * (kBytes + 16);
};

// Increments of the eight streamed populations over the node's own.  The
// gather of group q + 1 goes out member by member as group q is used up.
// LINK: a direction that is a link takes the reflected population at its own
// point x + t s e_k (t = tt[k-1] = 1 - 2q), from the same rows: with x = t e
// the weight is m0 (1 - t^2) + t^2 U +- t m1 (and V, W, W' in turn).
template <int KQ, bool LINK, class WaitM>
__device__ __forceinline__ void wls_increments(const float4* __restrict__ f8in, const float4* base, const int4* id,
                                               const float4& oa, const float4& ob, uint32_t mask, const float* tt,
                                               float* acc, WaitM wait_m) {
    constexpr int kSp = TileRec<KQ>::kSp;
    float4 ga[4], gb[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) ldg_pair_now(f8in + 2 * (size_t)at4(id[0], c), ga[c], gb[c]);
    wait_m();
#pragma unroll
    for (int q = 0; q < KQ; ++q) {
        float4 m[6];
        slot_rows<KQ>(base, q, m);
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
            if (q + 1 < KQ && !(q + 1 == kSp && c == 3))
                ldg_pair_now(f8in + 2 * (size_t)at4(id[(q + 1) % KQ], c), ga[c], gb[c]);
        }
    }
}

// the new state of a node that other partitions reference, into their halo slots
__device__ __forceinline__ void send_state(const PartDev* parts, const PartDev& own, int parity, int p, const float4& a,
                                           const float4* b) {
    const int e1 = own.send_first[p + 1];
    for (int e = own.send_first[p]; e < e1; ++e) {
        const int2 to = own.sends[e];
        float4* dst = parts[to.x].state[parity];
        if (b) {
            dst[2 * (size_t)to.y] = a;
            dst[2 * (size_t)to.y + 1] = *b;
        } else {
            dst[to.y] = a;
        }
    }
}

// One block's walk over range `rb` of the tiles.  PART: a partition of a
// partitioned set (own, one of parts), whose new states go to buffer `parity`
// of the partitions that hold them as halo.
template <int KQ, int MODEL, int WARPS, bool PART>
__device__ __forceinline__ void walk_tiles(const Stencil& S, const float4* __restrict__ in,
                                           const float* __restrict__ f0in, float4* __restrict__ out,
                                           float* __restrict__ f0out, const Collide& C0, int rb, int backward,
                                           int* __restrict__ err, const Wait& W, const PartDev* parts,
                                           const PartDev* own, int parity) {
    using L = WarpTile<KQ, WARPS>;
    using R = TileRec<KQ>;
    extern __shared__ __align__(128) uint8_t smem[];
    const int warp = threadIdx.x >> 5;
    const unsigned lane = threadIdx.x & 31u;
    uint8_t* slot = smem + warp * L::kBytes;
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + L::kWarps * L::kBytes) + 2 * warp;
    const float4* base = reinterpret_cast<const float4*>(slot) + lane;
    const int t0 = S.range[rb], t1 = S.range[rb + 1];
    if (warp >= t1 - t0) return;
    int t = backward ? t1 - 1 - warp : t0 + warp;
    const int hop = backward ? -L::kWarps : L::kWarps;
    // lane 0: index rows of a tile (need 0: only the row with the kind word), then its matrix rows
    int need_next = 0;
    auto copy_idx = [&](int tile) {
        const uint8_t* src = reinterpret_cast<const uint8_t*>(S.rec) + (size_t)tile * L::kBytes;
        if (need_next == 0) {
            mbar_expect_tx(bar, 512);
            bulk_g2s(slot + R::kSp * 512, src + R::kSp * 512, 512, bar);
        } else {
            const uint32_t bytes = need_next == 1 ? 3 * 512 : KQ * 512;
            mbar_expect_tx(bar, bytes);
            bulk_g2s(slot, src, bytes, bar);
        }
    };
    auto copy_m = [&](int tile) {
        if (need_next != 2) return;
        const uint8_t* src = reinterpret_cast<const uint8_t*>(S.rec) + (size_t)tile * L::kBytes;
        mbar_expect_tx(bar + 1, L::kBytes - KQ * 512);
        bulk_g2s(slot + KQ * 512, src + KQ * 512, L::kBytes - KQ * 512, bar + 1);
    };
    bool withhold = W.withhold && blockIdx.x == 0 && warp == 0;
    if (lane == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 1, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        need_next = S.need[t];
        if (!withhold) {
            copy_idx(t);
            copy_m(t);
        }
    }
    __syncwarp();
    pdl_trigger();
    pdl_wait();
    uint32_t ph = 0, phm = 0;
    for (; t >= t0 && t < t1; t += hop) {
        const int tn = t + hop;
        const int need = __shfl_sync(0xffffffffu, need_next, 0);
        const int p = t * 32 + (int)lane;
        const bool last = tn < t0 || tn >= t1;
        bool ok = __all_sync(0xffffffffu, mbar_wait(bar, ph, W.budget_ns));
        if (!ok) {
            if (lane == 0) {
                atomicExch(err, 2);
                // do not leave while copies may still be landing
                if (!withhold) mbar_wait(bar, ph, W.budget_ns);
                if (need == 2 && !withhold) mbar_wait(bar + 1, phm, W.budget_ns);
            }
            return;
        }
        ph ^= 1u;
        int4 id[KQ];
#pragma unroll
        for (int q = 0; q < KQ; ++q) id[q] = reinterpret_cast<const int4*>(base)[q * 32];
        __syncwarp();
        if (lane == 0 && !last) {
            need_next = S.need[tn];
            copy_idx(tn);
        }
        const int word = id[R::kSp].w;
        const uint8_t meta = (uint8_t)(word & 0xff);
        const int kind = meta & 3;
        bool m_ok = true;
        auto wait_m = [&]() { m_ok = mbar_wait(bar + 1, phm, W.budget_ns); };
        auto m_done = [&]() {
            // the slot's matrix rows are read: refill them for the warp's next tile
            if (need == 2) {
                m_ok = __all_sync(0xffffffffu, m_ok && mbar_wait(bar + 1, phm, W.budget_ns));
                if (!m_ok) return false;
                phm ^= 1u;
            }
            // the vote above orders no memory: every lane's reads come before the copy over them by this
            __syncwarp();
            if (lane == 0 && !last) copy_m(tn);
            return true;
        };
        const Collide C = S.coll ? S.coll[word >> 8] : C0;
        if (MODEL == 0) {
            float4 oa = make_float4(0, 0, 0, 0), ob = oa;
            float f0own = 0.f;
            float acc[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] = 0.f;
            LinkRec lk;
            lk.mask = 0;
            const bool links = (meta & 4) && kind != 2;
            if (kind != 2) {
                ldg_pair_now(in + 2 * (size_t)p, oa, ob);
                f0own = f0in[p];
            }
            if (links) lk = S.links[S.link_slot[p]];
            const bool moved = S.bb_mode != 0 && __any_sync(0xffffffffu, links && kind == 0);
            if (kind == 0) {
                if (moved) {
                    float tt[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) tt[k] = ((lk.mask >> (k + 1)) & 1u) ? lk.t[k] : -1.0f;
                    wls_increments<KQ, true>(in, base, id, oa, ob, lk.mask, tt, acc, wait_m);
                } else {
                    wls_increments<KQ, false>(in, base, id, oa, ob, 0u, nullptr, acc, wait_m);
                }
            }
            if (!m_done()) {
                if (lane == 0) {
                    atomicExch(err, 2);
                    // do not leave while copies may still be landing
                    if (!last) mbar_wait(bar, ph, W.budget_ns);
                    mbar_wait(bar + 1, phm, W.budget_ns);
                }
                return;
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
                    const int ids[9] = {id[0].x, id[0].y, id[0].z, id[0].w, id[1].x, id[1].y, id[1].z, id[1].w,
                                        id[2].x};
                    const float r = __int_as_float(id[2].y), cx = (float)ex_of(meta >> 4),
                                cy = (float)ey_of(meta >> 4);
                    lagrange_increments<1>([&](int j, float4& a, float4& b) { ldg_pair(in + 2 * (size_t)j, a, b); },
                                           ids, r, cx, cy, oa, ob, 0, acc);
#pragma unroll
                    for (int k = 0; k < 8; ++k) g[k + 1] = acc[k] + own[k];
                    if (links)
#pragma unroll
                        for (int k = 1; k < 9; ++k) {
                            if (!((lk.mask >> k) & 1u)) continue;
                            const int kp = opp_of(k);
                            g[k] = S.bb_mode == 0 ? own[kp - 1]
                                                  : lagrange_link([&](int j, int kk) { return pop(in, j, kk); }, ids, r,
                                                                  cx, cy, k, lk.t[k - 1], own[kp - 1]);
                        }
                }
                g[0] = f0own;
                collide_pairs(g, C, 0xFu, true);
            }
            if (p < S.n) {
                out[2 * (size_t)p] = make_float4(g[1], g[2], g[3], g[4]);
                out[2 * (size_t)p + 1] = make_float4(g[5], g[6], g[7], g[8]);
                f0out[p] = g[0];
                if (PART && (meta & 8)) {
                    const float4 hi = make_float4(g[5], g[6], g[7], g[8]);
                    send_state(parts, *own, parity, p, make_float4(g[1], g[2], g[3], g[4]), &hi);
                }
            }
        } else {
            float4 me = make_float4(0, 0, 0, 0);
            if (kind != 2) me = ldg_now(in + p);
            float c[3][6];
#pragma unroll
            for (int f = 0; f < 3; ++f)
#pragma unroll
                for (int a = 0; a < 6; ++a) c[f][a] = 0.f;
            float4 v9[9];
            if (kind == 0) {
                float4 nb[4 * KQ];
#pragma unroll
                for (int j = 0; j < 4 * KQ; ++j)
                    if (j != 4 * R::kSp + 3) nb[j] = ldg_now(in + at4(id[j / 4], j % 4));
                wait_m();
#pragma unroll
                for (int q = 0; q < KQ; ++q) {
                    float4 m[6];
                    slot_rows<KQ>(base, q, m);
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc) {
                        if (q == R::kSp && cc == 3) continue;
                        const float4 rv = nb[4 * q + cc];
                        const float vx = rv.x - me.x, vy = rv.y - me.y, vz = rv.z - me.z;
#pragma unroll
                        for (int a = 0; a < 6; ++a) {
                            const float ma = at4(m[a], cc);
                            c[0][a] = fmaf(ma, vx, c[0][a]);
                            c[1][a] = fmaf(ma, vy, c[1][a]);
                            c[2][a] = fmaf(ma, vz, c[2][a]);
                        }
                    }
                }
            }
            if (!m_done()) {
                if (lane == 0) {
                    atomicExch(err, 2);
                    // do not leave while copies may still be landing
                    if (!last) mbar_wait(bar, ph, W.budget_ns);
                    mbar_wait(bar + 1, phm, W.budget_ns);
                }
                return;
            }
            if (kind == 2) {
                if (p < S.n) {
                    out[p] = S.eqv[p];
                    if (PART && (meta & 8)) send_state(parts, *own, parity, p, S.eqv[p], nullptr);
                }
            } else {
                float r = 0.f, cx = 0.f, cy = 0.f;
                if (kind == 0) {
#pragma unroll
                    for (int f = 0; f < 3; ++f) {
                        float tc[6];
#pragma unroll
                        for (int a = 0; a < 6; ++a) tc[a] = c[f][a];
                        unbasis(tc, c[f]);
                    }
                } else if constexpr (KQ >= 3) {
                    const int ids[9] = {id[0].x, id[0].y, id[0].z, id[0].w, id[1].x, id[1].y, id[1].z, id[1].w,
                                        id[2].x};
#pragma unroll
                    for (int b = 0; b < 9; ++b) v9[b] = ldg_now(in + ids[b]);
                    r = __int_as_float(id[2].y);
                    cx = (float)ex_of(meta >> 4);
                    cy = (float)ey_of(meta >> 4);
                }
                const float4 o = tau1_finish(S, C, me, kind, c, v9, r, cx, cy, links_of(S, p, (meta & 4) != 0));
                if (p < S.n) {
                    out[p] = o;
                    if (PART && (meta & 8)) send_state(parts, *own, parity, p, o, nullptr);
                }
            }
        }
    }
}

template <int KQ, int MODEL, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 1)
    step_warp(Stencil S, const float4* __restrict__ in, const float* __restrict__ f0in, float4* __restrict__ out,
              float* __restrict__ f0out, Collide C0, int backward, int* __restrict__ err, const Wait W) {
    walk_tiles<KQ, MODEL, WARPS, false>(S, in, f0in, out, f0out, C0, blockIdx.x, backward, err, W, nullptr, nullptr,
                                        0);
}

// All partitions of a partitioned set in one launch: block b walks range
// work[b].y of partition work[b].x, from buffer `from` into the other one.
template <int KQ, int MODEL, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 1)
    step_parts(const PartDev* __restrict__ parts, const int2* __restrict__ work, int from, int backward,
               int* __restrict__ err, const Wait W) {
    const int2 job = work[blockIdx.x];
    const PartDev* own = parts + job.x;
    const Stencil S = own->S;
    const Collide C0 = own->C;
    walk_tiles<KQ, MODEL, WARPS, true>(S, own->state[from], own->f0[from], own->state[from ^ 1], own->f0[from ^ 1], C0,
                                       job.y, backward, err, W, parts, own, from ^ 1);
}

// bit 3 of the kind bytes (and the records' copies) of nodes whose states are sent
__global__ void mark_sends(int n, const int* __restrict__ send_first, uint8_t* __restrict__ meta) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n && send_first[p + 1] > send_first[p]) meta[p] |= 8;
}

// Halo copies of all partitions, w float4 a state: entry (owner, its position,
// receiver, its slot).
__global__ void exchange_states(const PartDev* __restrict__ parts, const int4* __restrict__ list, int64_t m, int w,
                                int cur) {
    const int64_t total = m * w;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int4 e = list[i / w];
        const size_t c = (size_t)(i % w);
        parts[e.z].state[cur][(size_t)e.w * w + c] = parts[e.x].state[cur][(size_t)e.y * w + c];
    }
}

// The tile records' copies of the kind bytes, and what each tile has to fetch,
// after kinds have changed.  The next step kernel reads both before it waits
// for its predecessor, so the stream is synchronised in between.
__global__ void record_kinds(int n, int rows, int sp, const uint8_t* __restrict__ meta, int4* __restrict__ rec,
                             uint8_t* __restrict__ need) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = p & 31, tile = p >> 5;
    int kind = 2;
    if (p < n) {
        const uint8_t t = meta[p];
        kind = t & 3;
        int& word = rec[((size_t)tile * rows + sp) * 32 + lane].w;
        word = (word & ~0xff) | t;
    }
    const bool any0 = __any_sync(0xffffffffu, kind == 0), any1 = __any_sync(0xffffffffu, kind == 1);
    if (lane == 0 && tile * 32 < n) need[tile] = any0 ? 2 : (any1 ? 1 : 0);
}

// Cuts the tiles into n_ranges contiguous ranges of about equal cost (one
// block): every thread adds up a run of tiles, the block scans the sums, and
// each thread sets the range starts that fall into its run.
__global__ void __launch_bounds__(1024) tile_ranges(int n_tiles, const uint8_t* __restrict__ need, int n_ranges,
                                                    int* __restrict__ range) {
    __shared__ long long sum[1024];
    const int tid = threadIdx.x;
    const int a = (int)((int64_t)n_tiles * tid / 1024), b = (int)((int64_t)n_tiles * (tid + 1) / 1024);
    auto cost = [&](int t) { return need[t] == 2 ? kCostStencil : (need[t] == 1 ? kCostLagrange : kCostCopy); };
    long long own = 0;
    for (int t = a; t < b; ++t) own += cost(t);
    sum[tid] = own;
    __syncthreads();
    for (int h = 1; h < 1024; h *= 2) {
        const long long v = tid >= h ? sum[tid - h] : 0;
        __syncthreads();
        sum[tid] += v;
        __syncthreads();
    }
    const long long total = sum[1023];
    long long before = sum[tid] - own;
    for (int t = a; t < b; ++t) {
        const long long after = before + cost(t);
        for (long long r = (before * n_ranges + total - 1) / total; r * total < after * n_ranges; ++r)
            range[r] = t;
        before = after;
    }
    if (tid == 0) range[n_ranges] = n_tiles;
}

}  // namespace dev

namespace {

// Bytes of records above which steps walk back over what the last one left in
// L2.  Below ~100 MB everything stays there and the order is worth nothing
// (192k nodes, 83 MB: 14.3 us forwards, 14.6 in turn); above it every step
// saves what L2 holds (260k nodes, 112 MB: 22.9 -> 20.4 us; 420k tau = 1: 33.0
// -> 30.1 us; 1.73M: 122.9 -> 120.1 us).
constexpr size_t kResident = size_t(100) << 20;

template <int KQ, int MODEL, int WARPS>
cudaError_t run_warp(const dev::Stencil& S, const float4* in, const float* f0in, float4* out, float* f0out,
                     const dev::Collide& C, int backward, int* err, const dev::Wait& W, cudaStream_t st) {
    using L = dev::WarpTile<KQ, WARPS>;
    static_assert(L::kSmem <= 232448, "slots exceed shared memory");
    auto fn = dev::step_warp<KQ, MODEL, WARPS>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kSmem);
    if (e != cudaSuccess) return e;
    const int back = (size_t)((S.n + 31) / 32) * L::kBytes > kResident ? backward : 0;
    return launch_pdl_smem(fn, S.n_ranges, WARPS * 32, L::kSmem, st, S, in, f0in, out, f0out, C, back, err, W);
}

template <int KQ, int WARPS>
cudaError_t run_warp_model(int model, const dev::Stencil& S, const float4* a8, const float* a0, float4* b8, float* b0,
                           const float4* ra, float4* rb, const dev::Collide& C, int backward, int* err,
                           const dev::Wait& W, cudaStream_t st) {
    return model == 0 ? run_warp<KQ, 0, WARPS>(S, a8, a0, b8, b0, C, backward, err, W, st)
                      : run_warp<KQ, 1, WARPS>(S, ra, a0, rb, b0, C, backward, err, W, st);
}

// slots per block: variant 27 as many as leave the registers and L1 the
// gathers need, 28 fewer, 29 as many as fit or register counts allow
template <int KQ, int W27, int W28, int W29>
cudaError_t run_warp_variant(int variant, int model, const dev::Stencil& S, const float4* a8, const float* a0,
                             float4* b8, float* b0, const float4* ra, float4* rb, const dev::Collide& C, int backward,
                             int* err, const dev::Wait& W, cudaStream_t st) {
    switch (variant) {
        case 27: return run_warp_model<KQ, W27>(model, S, a8, a0, b8, b0, ra, rb, C, backward, err, W, st);
        case 28: return run_warp_model<KQ, W28>(model, S, a8, a0, b8, b0, ra, rb, C, backward, err, W, st);
        case 29: return run_warp_model<KQ, W29>(model, S, a8, a0, b8, b0, ra, rb, C, backward, err, W, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_step_warp(int variant, int model, const dev::Stencil& S, const float4* a8, const float* a0,
                             float4* b8, float* b0, const float4* ra, float4* rb, const dev::Collide& C, int backward,
                             int* err, const dev::Wait& W, cudaStream_t st) {
    if (S.n == 0) return cudaSuccess;
    switch (S.Kq) {
        case 3: return run_warp_variant<3, 12, 8, 14>(variant, model, S, a8, a0, b8, b0, ra, rb, C, backward, err, W, st);
        case 4: return run_warp_variant<4, 12, 8, 14>(variant, model, S, a8, a0, b8, b0, ra, rb, C, backward, err, W, st);
        case 6: return run_warp_variant<6, 10, 8, 11>(variant, model, S, a8, a0, b8, b0, ra, rb, C, backward, err, W, st);
        case 8: return run_warp_variant<8, 8, 6, 7>(variant, model, S, a8, a0, b8, b0, ra, rb, C, backward, err, W, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_step_parts(int model, int Kq, int64_t n, const dev::PartDev* parts, const int2* work, int blocks,
                              int from, int* err, const dev::Wait& W, cudaStream_t st) {
    const int back = (size_t)(n / 32) * (7 * Kq - 1) * 512 > kResident ? from : 0;
    auto run = [&](auto fn, int warps, size_t smem) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        return launch_pdl_smem(fn, blocks, warps * 32, smem, st, parts, work, from, back, err, W);
    };
#define MLBM_PARTS(KQ, WARPS)                                                                              \
    case KQ:                                                                                               \
        return model == 0 ? run(dev::step_parts<KQ, 0, WARPS>, WARPS, dev::WarpTile<KQ, WARPS>::kSmem)     \
                          : run(dev::step_parts<KQ, 1, WARPS>, WARPS, dev::WarpTile<KQ, WARPS>::kSmem);
    switch (Kq) {
        MLBM_PARTS(3, 12)
        MLBM_PARTS(4, 12)
        MLBM_PARTS(6, 10)
        MLBM_PARTS(8, 8)
        default: return cudaErrorInvalidValue;
    }
#undef MLBM_PARTS
}

cudaError_t launch_mark_sends(int n, const int* send_first, uint8_t* meta, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    dev::mark_sends<<<(n + 255) / 256, 256, 0, st>>>(n, send_first, meta);
    return cudaGetLastError();
}

cudaError_t launch_exchange(const dev::PartDev* parts, const int4* list, int64_t m, int w, int cur, cudaStream_t st) {
    if (m == 0) return cudaSuccess;
    const int grid = (int)std::min<int64_t>(8 * 152, (m * w + 255) / 256);
    dev::exchange_states<<<grid, 256, 0, st>>>(parts, list, m, w, cur);
    return cudaGetLastError();
}

int warp_step_ranges(int n) {
    int dev_id = 0, sms = 0;
    cudaGetDevice(&dev_id);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev_id);
    return std::max(1, std::min((n + 31) / 32, sms));
}

cudaError_t launch_record_kinds(const dev::Stencil& S, float4* rec, uint8_t* need, int* range, cudaStream_t st) {
    if (!rec || S.n == 0) return cudaSuccess;
    dev::record_kinds<<<(S.n + 255) / 256, 256, 0, st>>>(S.n, S.rows, dev::special_group(S.Kq), S.meta,
                                                         reinterpret_cast<int4*>(rec), need);
    dev::tile_ranges<<<1, 1024, 0, st>>>((S.n + 31) / 32, need, S.n_ranges, range);
    return cudaGetLastError();
}

}  // namespace mlbm
