// C-ABI glue: simulation contexts, state I/O, the step loop and observables.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <memory>
#include <string>
#include <vector>

#include "kernels.h"
#include "mlbm_internal.h"

namespace mlbm {

thread_local std::string g_last_error;

mlbm_status set_error(mlbm_status st, const std::string& msg) {
    g_last_error = msg;
    return st;
}
void clear_error() { g_last_error.clear(); }

}  // namespace mlbm

using namespace mlbm;

struct mlbm_ctx {
    int device = 0;
    mlbm_params params{};
    int64_t n = 0, n_pad = 0;
    int64_t n_halo = 0;  // state slots after the n nodes (partitions only)
    int K = 0;
    double s = 1.0, box_area = 1.0;
    cudaStream_t stream = nullptr;
    cudaStream_t own_stream = nullptr;
    // stencil data on the device
    float4* rec = nullptr;    // tile records (see dev::TileRec; least-squares stencils)
    uint8_t* need = nullptr;  // what each tile fetches of its record
    int* range = nullptr;     // tile ranges of the step's blocks
    int4* idx = nullptr;      // RBF-FD stencils
    uint8_t* meta = nullptr;
    float* lag_r = nullptr;
    int* link_slot = nullptr;
    dev::LinkRec* links = nullptr;
    float4* eqv = nullptr;
    int* perm = nullptr;
    float* area = nullptr;
    float* area_over_s2 = nullptr;
    uint8_t* mask = nullptr;
    int* link_nodes = nullptr;
    int n_link_nodes = 0;
    // state
    float4* f8[2] = {nullptr, nullptr};
    float* f0[2] = {nullptr, nullptr};
    float4* ruv[2] = {nullptr, nullptr};
    int cur = 0;
    // work
    float *rho = nullptr, *px = nullptr, *py = nullptr;
    double* io = nullptr;
    double* scratch = nullptr;
    int64_t scratch_len = 0;
    int64_t steps = 0;
    int64_t steps_in_last_run = 0;  // steps taken by the last run to steady state
    bool timing = false;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    double last_ms = -1.0;
    int variant = 27;
    std::vector<int> inv_perm;  // caller's node id -> device position
    int* err = nullptr;  // device error word of the bounded waits
    bool rbf_tiles_default = false;  // large sets: every plain capped number steps from RBF-FD tile records
    int cluster = 0;  // blocks of the cluster that takes runs of steps (0: the set does not fit one)
    dev::Stencil S{};
    dev::Collide C{};
    std::vector<void*> allocations;
    // batch of independent samples (empty for a single sample)
    std::vector<int64_t> seg_off;  // position offset of each sample, plus the total
    std::vector<mlbm_params> seg_params;
    std::vector<double> seg_box_area;
    std::vector<double> seg_s;  // streaming distance of each sample
    // device: the error word of the bounded waits (err, 8 bytes) and behind it
    // the results of an observable, up to 9 doubles per sample, so that one
    // copy brings both back
    double* seg_out = nullptr;
    int64_t* seg_dev = nullptr;  // seg_off on the device
    int max_blocks = 1;          // reduction blocks of the largest sample
    std::vector<int> link_off;   // first link node of each sample, plus the total
    // captured step graphs: chunk of kGraphSteps steps starting from buffer 0 / 1
    bool use_graphs = true;
    cudaGraphExec_t graph[2] = {nullptr, nullptr};
    int graph_variant = -1;
    cudaStream_t graph_stream = nullptr;
    // bounded waits of the bulk-copy variants (4..7, 27..29): budget of one wait,
    // and the test switch that makes the next launch withhold one tile
    unsigned long long wait_ns = 2000000000ULL;
    int withhold_next = 0;
    // device buffer of mlbm_wall_stress_force, grown on demand and kept:
    // positions, normals, lengths and tractions of up to wall_cap wall nodes
    uint8_t* wall_buf = nullptr;
    int64_t wall_cap = 0;
    // per-step time of every variant in the last autotune (-1: not timed)
    std::vector<double> tune_ms;
};

namespace {
constexpr int kGraphSteps = 16;
constexpr int kMaxK = 64;  // widest device stencil (RBF-FD unions per Lagrangian point)
constexpr int kMaxVariant = 29;  // step kernel variants 0..29 (see mlbm_set_kernel_variant)
}

// Cold-cache start for timed steps: reading a zeroed buffer several times the
// size of L2 leaves L2 holding clean lines of that buffer only, so a timed
// step neither hits its own data nor pays for writing back dirty lines left
// by whatever ran before (which a memset flush would leave behind).
__global__ void l2_flush_read(const float4* __restrict__ buf, size_t n, float* sink) {
    float acc = 0.f;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float4 v = __ldcg(buf + i);
        acc += (v.x + v.y) + (v.z + v.w);
    }
    if (acc != 0.f) *sink = acc;  // never taken on the zeroed buffer; keeps the loads
}

namespace {

#define MLBM_CUDA(call)                                                                                      \
    do {                                                                                                     \
        cudaError_t e_ = (call);                                                                             \
        if (e_ != cudaSuccess)                                                                               \
            return set_error(MLBM_E_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));               \
    } while (0)

template <class T>
mlbm_status dalloc(mlbm_ctx* c, T** p, size_t count) {
    void* q = nullptr;
    cudaError_t e = cudaMalloc(&q, std::max<size_t>(count, 1) * sizeof(T));
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return set_error(e == cudaErrorMemoryAllocation ? MLBM_E_OOM : MLBM_E_CUDA,
                         std::string("cudaMalloc: ") + cudaGetErrorString(e));
    }
    c->allocations.push_back(q);
    *p = static_cast<T*>(q);
    return MLBM_OK;
}

#define MLBM_TRY(expr)                       \
    do {                                     \
        mlbm_status s_ = (expr);             \
        if (s_ != MLBM_OK) return s_;        \
    } while (0)

mlbm_status upload(mlbm_ctx* c, void* dst, const void* src, size_t bytes) {
    MLBM_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, c->stream));
    return MLBM_OK;
}

void set_collide(mlbm_ctx* c) {
    const double tp = c->params.tau;
    const double tm = c->params.tau_minus > 0 ? c->params.tau_minus : tp;
    c->C.omega_p = (float)(1.0 / tp);
    c->C.omega_m = (float)(1.0 / tm);
    c->C.src_p = (float)(1.0 - 0.5 / tp);
    c->C.src_m = (float)(1.0 - 0.5 / tm);
    c->C.ax = (float)c->params.gx;
    c->C.ay = (float)c->params.gy;
}

mlbm_status check_params(const mlbm_params* p) {
    if (p->model != MLBM_MODEL_BGK && p->model != MLBM_MODEL_TAU1) return set_error(MLBM_E_INVALID, "bad model");
    if (!(p->tau > 0.5) || !std::isfinite(p->tau)) return set_error(MLBM_E_INVALID, "tau must be > 1/2");
    if (p->tau_minus > 0 && !(p->tau_minus > 0.5)) return set_error(MLBM_E_INVALID, "tau_minus must be > 1/2");
    if (p->model == MLBM_MODEL_TAU1 && (p->tau != 1.0 || (p->tau_minus > 0 && p->tau_minus != 1.0)))
        return set_error(MLBM_E_INVALID, "the tau = 1 model needs tau = tau_minus = 1");
    if (!std::isfinite(p->gx) || !std::isfinite(p->gy)) return set_error(MLBM_E_INVALID, "non-finite body force");
    return MLBM_OK;
}

// a set error word: cleared in stream order, before any later launch can set
// it again, and reported
mlbm_status wait_failed(mlbm_ctx* c, int code) {
    MLBM_CUDA(cudaMemsetAsync(c->err, 0, sizeof(int), c->stream));
    MLBM_CUDA(cudaStreamSynchronize(c->stream));
    return set_error(MLBM_E_TIMEOUT, "a bounded device wait gave up (code " + std::to_string(code) +
                                         "); the step result is invalid");
}

mlbm_status sync(mlbm_ctx* c) {
    int e = 0;
    if (c->err) MLBM_CUDA(cudaMemcpyAsync(&e, c->err, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    MLBM_CUDA(cudaStreamSynchronize(c->stream));
    return e != 0 ? wait_failed(c, e) : MLBM_OK;
}

// the first `count` results and the error word, in one copy
mlbm_status read_results(mlbm_ctx* c, double* h, size_t count) {
    std::vector<double> buf(count + 1);
    const bool together = reinterpret_cast<double*>(c->err) + 1 == c->seg_out;
    if (together) {
        MLBM_CUDA(cudaMemcpyAsync(buf.data(), c->err, (count + 1) * 8, cudaMemcpyDeviceToHost, c->stream));
        MLBM_CUDA(cudaStreamSynchronize(c->stream));
        int e = 0;
        std::memcpy(&e, buf.data(), sizeof(int));
        if (e != 0) return wait_failed(c, e);
    } else {  // a partition, whose error word lies elsewhere
        MLBM_CUDA(cudaMemcpyAsync(buf.data() + 1, c->seg_out, count * 8, cudaMemcpyDeviceToHost, c->stream));
        MLBM_TRY(sync(c));
    }
    std::copy(buf.begin() + 1, buf.end(), h);
    return MLBM_OK;
}

// whether a number steps from RBF-FD tile records, which exist where any does
bool by_rbf_tiles(const mlbm_ctx* c, int variant) {
    if (!c->S.rbf_rec) return false;
    if (variant == 28 || variant == 29) return true;
    // the numbers that run the plain capped kernel
    return c->rbf_tiles_default && variant != 0 && variant != 10 && variant != 12 && variant != 20 && variant != 21;
}

mlbm_status launch_one_step(mlbm_ctx* c, int variant) {
    const int a = c->cur, b = c->cur ^ 1;
    const int model = c->params.model == MLBM_MODEL_BGK ? 0 : 1;
    if (((variant >= 4 && variant <= 7) || (variant >= 27 && variant <= 29)) && !c->S.Wr) {
        const dev::Wait W{c->wait_ns, c->withhold_next};
        c->withhold_next = 0;
        if (variant <= 7)
            MLBM_CUDA(launch_step_tma(variant, model, c->S, c->f8[a], c->f0[a], c->f8[b], c->f0[b], c->ruv[a],
                                      c->ruv[b], c->C, c->err, W, c->stream));
        else  // every other step walks the tiles backwards
            MLBM_CUDA(launch_step_warp(variant, model, c->S, c->f8[a], c->f0[a], c->f8[b], c->f0[b], c->ruv[a],
                                       c->ruv[b], c->C, a, c->err, W, c->stream));
    }
    else if (model == 0 && by_rbf_tiles(c, variant))
        MLBM_CUDA(launch_step_rbf_tiles(c->S, c->f8[a], c->f0[a], c->f8[b], c->f0[b], c->C, a, c->err,
                                        dev::Wait{c->wait_ns, 0}, c->stream));
    else if (model == 0)
        MLBM_CUDA(launch_bgk_step(c->S, c->f8[a], c->f0[a], c->f8[b], c->f0[b], c->C, variant, c->stream));
    else
        MLBM_CUDA(launch_tau1_step(c->S, c->ruv[a], c->ruv[b], c->C, variant, c->stream));
    c->cur = b;
    return MLBM_OK;
}

// Runs of at least this many steps go to the cluster kernel where the set fits
// it; a shorter one does not repay the fetch of all records and states (us a
// call and wait, launches / cluster, 2000 nodes: 4 steps 22.6 / 24.7, 6 steps
// 29.1 / 28.9, 8 steps 35.2 / 32.9, 12 steps 47.1 / 42.0; 500 nodes: 22.9 / 21.9,
// 29.2 / 25.8, 34.7 / 29.3, 47.0 / 35.9).
constexpr int kClusterMin = 8;
constexpr int kClusterSteps = 4096;  // most steps of one launch

bool by_cluster(const mlbm_ctx* c, int64_t n_steps, int variant) {
    return c->cluster > 0 && variant == 27 && c->use_graphs && n_steps >= kClusterMin;
}

mlbm_status launch_cluster_steps(mlbm_ctx* c, int64_t n_steps) {
    for (int64_t left = n_steps; left > 0;) {
        const int m = (int)std::min<int64_t>(left, kClusterSteps), a = c->cur, b = a ^ (m & 1);
        const dev::Wait W{c->wait_ns, c->withhold_next};
        c->withhold_next = 0;
        MLBM_CUDA(launch_step_cluster(c->cluster, c->S, c->f8[a], c->f0[a], c->f8[b], c->f0[b], c->C, m, c->err, W,
                                      c->stream));
        c->cur = b;
        left -= m;
    }
    return MLBM_OK;
}

// A BGK context of RBF-FD stencils steps from tile records of its non-zero weights
// where the plain rows (36 K bytes a node) take more than 60 MB and the records at
// most two thirds of that.  From about 55 MB on, the plain step depends on where
// the rows happen to lie in L2: the same set took up to 40% longer in one process
// than in another, while the records, of half the size, always took the same.  us a
// step, plain least .. median .. most of eight processes / records:
//   K = 64, 25 nodes a point: 38 MB 9.5 .. 9.6 .. 9.6 / 6.6, 55 MB 9.8 .. 11.4 ..
//   12.5 / 9.6, 66 MB 10.2 .. 14.2 .. 14.7 / 11.9, 79 MB 12.5 .. 16.0 .. 16.4 /
//   11.9, 87 MB 14.4 .. 17.6 .. 18.0 / 12.6; 150 MB 25.4 / 18.8
//   K = 48, 15 nodes: 54 MB 8.2 / 9.6, 59 MB 8.7 / 10.0, 73 MB 13.0 .. 14.4 .. 14.9 / 10.3
//   K = 32, 7 nodes: 39 MB 6.3 / 8.0, 64 MB 9.8 .. 10.9 .. 11.1 / 9.4, 75 MB 10.6 ..
//   12.3 .. 13.3 / 11.6, 88 MB 12.7 .. 15.2 .. 15.5 / 12.1
// Below the line the winner changes with K.  Stencils of the node's own 24 have no
// zeros to leave out: 147k nodes 23.1 / 26.7, 260k 41.1 / 44.5.  Kernel variants 28
// and 29 take the records in any case, and only they where the rule does not make
// them the default.
constexpr size_t kRbfTilesFrom = 60000000;

// Releases the records (no step that reads them may be in flight).
void drop_rbf_tiles(mlbm_ctx* c) {
    for (const void* p : {(const void*)c->S.rbf_rec, (const void*)c->S.rbf_head, (const void*)c->S.rbf_range}) {
        c->allocations.erase(std::find(c->allocations.begin(), c->allocations.end(), p));
        cudaFree(const_cast<void*>(p));
    }
    c->S.rbf_rec = nullptr;
    c->S.rbf_head = nullptr;
    c->S.rbf_range = nullptr;
}

// The records of the RBF-FD step from the uploaded stencils.  Where they do
// not fit (node numbers of 28 bits, no memory) the context steps without them.
mlbm_status build_rbf_tiles(mlbm_ctx* c, bool always) {
    const int tiles = (int)((c->n + 15) / 16);
    if (tiles == 0 || c->n + c->n_halo >= (int64_t)1 << 28) return MLBM_OK;
    std::vector<void*> made;
    auto room = [&](void** p, size_t bytes) {
        if (cudaMalloc(p, std::max<size_t>(bytes, 128)) != cudaSuccess) {
            (void)cudaGetLastError();
            for (void* q : made) cudaFree(q);
            return false;
        }
        made.push_back(*p);
        return true;
    };
    void *dsize = nullptr, *drec = nullptr, *dhead = nullptr, *drange = nullptr;
    if (!room(&dsize, (size_t)tiles * sizeof(int2))) return MLBM_OK;
    std::vector<int2> size((size_t)tiles);
    cudaError_t e = rbf_tile_sizes(c->S, tiles, static_cast<int2*>(dsize), c->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(size.data(), dsize, size.size() * sizeof(int2), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    cudaFree(dsize);
    made.clear();
    MLBM_CUDA(e);
    std::vector<int4> head;
    std::vector<int> range;
    const int blocks = std::min(tiles, warp_step_ranges(1 << 30));
    if (!rbf_tiles_plan(size, blocks, head, range, c->S.rbf_slot, c->S.rbf_bytes)) return MLBM_OK;
    if (!always && 3 * c->S.rbf_bytes > 2 * (size_t)c->n * 36 * c->K) return MLBM_OK;
    if (!room(&drec, c->S.rbf_bytes) || !room(&dhead, head.size() * sizeof(int4)) ||
        !room(&drange, range.size() * sizeof(int)))
        return MLBM_OK;
    for (void* q : made) c->allocations.push_back(q);
    MLBM_TRY(upload(c, dhead, head.data(), head.size() * sizeof(int4)));
    MLBM_TRY(upload(c, drange, range.data(), range.size() * sizeof(int)));
    MLBM_CUDA(rbf_tile_fill(c->S, tiles, static_cast<int4*>(dhead), static_cast<uint8_t*>(drec), c->stream));
    MLBM_CUDA(cudaStreamSynchronize(c->stream));
    c->S.rbf_rec = static_cast<uint8_t*>(drec);
    c->S.rbf_head = static_cast<int4*>(dhead);
    c->S.rbf_range = static_cast<int*>(drange);
    c->S.rbf_blocks = blocks;
    return MLBM_OK;
}

mlbm_status do_init(mlbm_ctx* c, const mlbm_stencils* st, const mlbm_params* p, const double* rho0, const double* u0) {
    const HostStencils& H = st->h;
    MLBM_CUDA(cudaGetDevice(&c->device));
    MLBM_CUDA(cudaStreamCreateWithFlags(&c->own_stream, cudaStreamNonBlocking));
    c->stream = c->own_stream;
    c->params = *p;
    c->n = H.n;
    c->K = H.K;
    c->s = H.s;
    c->box_area = H.box_area;
    c->n_pad = (H.n + 127) / 128 * 128;
    const int64_t n = H.n, np = c->n_pad;
    if (H.K < 4 || H.K > kMaxK || H.K % 4 != 0)
        return set_error(MLBM_E_INVALID, "init: stencil width must be a multiple of 4 in [4, 64]");
    // state slots: the nodes, then the halo copies of a partition's neighbours
    c->n_halo = H.n_halo;
    const int64_t nps = (H.n + H.n_halo + 127) / 128 * 128;
    const int K = H.K, Kq = K / 4;
    // ---- host-side device layout
    const bool rbf = H.interp != MLBM_INTERP_WLS;  // per-direction RBF-FD weights
    const int rows = 7 * Kq - 1, sp = dev::special_group(Kq);
    // (tile records: cleared on all cores, 81 MB at 185k nodes of K = 16, which one
    // core fills in 4.4 ms)
    const size_t tile_words = (size_t)rows * 128, n_words = rbf ? 0 : (size_t)(np / 32) * tile_words;
    const std::unique_ptr<int32_t[]> hrec(new int32_t[n_words]);
#pragma omp parallel for schedule(static, 128)
    for (int64_t t = 0; t < (rbf ? 0 : np / 32); ++t) std::fill_n(hrec.get() + (size_t)t * tile_words, tile_words, 0);
    std::vector<int32_t> hidx(rbf ? (size_t)Kq * np * 4 : 0, 0);
    std::vector<float> hW(rbf ? (size_t)8 * Kq * np * 4 : 0, 0.f);
    std::vector<uint8_t> hmeta(np, 0), hmask(np, 0);
    std::vector<float> hlag(np, 0.f), harea(np, 0.f), has2(np, 0.f);
    std::vector<int> hslot(np, -1), hperm(np, 0), hlinknodes;
    std::vector<dev::LinkRec> hlinks;
    std::vector<float4> heqv(np, make_float4(0, 0, 0, 0));
    // link records in node order: their slots first, then every node's rows
    // in parallel (each node writes only its own positions)
    for (int64_t q = 0; q < n; ++q)
        if (H.link_mask[q]) {
            hslot[q] = (int)hlinknodes.size();
            hlinknodes.push_back((int)q);
        }
    hlinks.resize(hlinknodes.size());
    const bool parts = !H.part_off.empty();
#pragma omp parallel for schedule(static, 4096)
    for (int64_t q = 0; q < n; ++q) {
        const uint8_t kind = H.kind[q];
        const uint16_t lm = H.link_mask[q];
        hmeta[q] = (uint8_t)(kind | (lm ? 4 : 0) | (H.center[q] << 4));
        hmask[q] = kind != kKindEq;
        hperm[q] = (int)H.perm[q];
        harea[q] = (float)H.area[q];
        const double sq = H.s_node.empty() ? H.s : H.s_node[q];
        has2[q] = (float)(H.area[q] / (sq * sq));
        // sample of a batch's node, and the node's lane in its tile record
        const int sample =
            parts ? (int)(std::upper_bound(H.part_off.begin(), H.part_off.end(), q) - H.part_off.begin()) - 1 : 0;
        int32_t* lane = rbf ? nullptr : hrec.get() + (size_t)(q / 32) * tile_words + (q % 32) * 4;
        if (!rbf) lane[sp * 128 + 3] = (int32_t)hmeta[q] | (sample << 8);
        if (kind == kKindWls) {
            // stencil slots in increasing node position: lanes of a warp that
            // gather slot j of consecutive (Hilbert-ordered) nodes then touch
            // nearby addresses; the matrix columns follow the same order
            int order[kMaxK];
            for (int j = 0; j < K; ++j) order[j] = j;
            if (H.slot_key.empty())
                std::sort(order, order + K,
                          [&](int a, int b) { return H.idx[(size_t)q * K + a] < H.idx[(size_t)q * K + b]; });
            else
                std::sort(order, order + K, [&](int a, int b) {
                    return H.slot_key[(size_t)q * K + a] < H.slot_key[(size_t)q * K + b];
                });
            // the node's matrix or RBF-FD weight rows: its own, or its sample's
            const double* Mq = nullptr;
            const double* Wq = nullptr;
            if (parts) {
                const size_t l = (size_t)(q - H.part_off[sample]);
                if (rbf) Wq = H.part_Wr[sample] + l * 8 * K;
                else Mq = H.part_M[sample] + l * 6 * K;
            } else if (rbf) {
                Wq = H.Wr.data() + (size_t)q * 8 * K;
            } else {
                Mq = H.M.data() + (size_t)q * 6 * K;
            }
            if (rbf)
                for (int jj = 0; jj < K; ++jj) {
                    const int j = order[jj];
                    hidx[(((size_t)(jj / 4)) * np + q) * 4 + (jj % 4)] = H.idx[(size_t)q * K + j];
                    for (int k = 0; k < 8; ++k)
                        hW[(((size_t)(k * Kq + jj / 4)) * np + q) * 4 + (jj % 4)] = (float)Wq[(size_t)k * K + j];
                }
            int slot = 0;
            for (int jj = 0; !rbf && jj < K; ++jj) {
                const int j = order[jj];
                const int32_t id = H.idx[(size_t)q * K + j];
                if (id == q) continue;  // its weight multiplies a zero difference
                if (slot == 4 * sp + 3) ++slot;
                double m[6];
                for (int a = 0; a < 6; ++a) m[a] = Mq[(size_t)a * K + j];
                // D2Q9 departure basis (see device_common.cuh), formed in FP64
                const double t[6] = {m[0] + m[3], m[0] + m[5], m[0] + m[3] + m[4] + m[5], m[0] + m[3] - m[4] + m[5],
                                     m[1], m[2]};
                const int g = slot / 4, cc = slot % 4, mr = Kq + 6 * g - (g > sp ? 1 : 0);
                lane[g * 128 + cc] = id;
                for (int a = 0; a < 6; ++a) {
                    const float v = (float)t[a];
                    std::memcpy(g == sp && a == 5 ? &lane[(mr + cc) * 128 + 3] : &lane[(mr + a) * 128 + cc], &v, 4);
                }
                ++slot;
            }
        } else if (kind == kKindLagrange) {
            for (int b = 0; b < 9; ++b) {
                const int j = H.lag_slot[(size_t)q * 9 + b];
                (rbf ? hidx[(((size_t)(b / 4)) * np + q) * 4 + (b % 4)] : lane[(b / 4) * 128 + (b % 4)]) =
                    H.idx[(size_t)q * K + j];
            }
            hlag[q] = (float)(sq / H.lag_h[q]);
            if (!rbf) std::memcpy(&lane[2 * 128 + 1], &hlag[q], 4);
        } else {
            heqv[q] = make_float4((float)(H.eqv[q * 3] - 1.0), (float)H.eqv[q * 3 + 1], (float)H.eqv[q * 3 + 2], 0.f);
        }
        if (lm) {
            dev::LinkRec r{};
            r.mask = lm;
            for (int k = 1; k < 9; ++k) r.t[k - 1] = (float)(1.0 - 2.0 * H.q[(size_t)q * 9 + k]);
            hlinks[(size_t)hslot[q]] = r;
        }
    }
    // lanes past the last node read as equilibrium nodes, which gather nothing
    for (int64_t q = n; !rbf && q < np; ++q)
        hrec[(size_t)(q / 32) * tile_words + (q % 32) * 4 + (size_t)sp * 128 + 3] = kKindEq;
    c->n_link_nodes = (int)hlinknodes.size();
    c->inv_perm.assign((size_t)n, -1);
    for (int64_t q = 0; q < n; ++q) c->inv_perm[(size_t)hperm[q]] = (int)q;
    // ---- neighbourhood staging (variant 22, least-squares BGK): per tile of
    // kStageTile nodes the sorted union of the stencil members of its
    // least-squares nodes without links, and each member's local index
    std::vector<uint16_t> hlidx;
    std::vector<int> hsoff, hsids;
    int stage_max = 0;
    if (p->model == MLBM_MODEL_BGK && !rbf && tma_supported(Kq)) {
        const int64_t T = dev::kStageTile, nt = (n + T - 1) / T;
        std::vector<std::vector<int>> lists((size_t)nt);
        hlidx.assign((size_t)Kq * np * 4, 0);
        auto lane_of = [&](int64_t q) { return hrec.get() + (size_t)(q / 32) * tile_words + (q % 32) * 4; };
#pragma omp parallel for schedule(dynamic, 8)
        for (int64_t b = 0; b < nt; ++b) {
            std::vector<int>& L = lists[(size_t)b];
            const int64_t q0 = b * T, q1 = std::min<int64_t>(n, q0 + T);
            for (int64_t q = q0; q < q1; ++q)
                if ((hmeta[q] & 7) == 0)
                    for (int g = 0; g < Kq; ++g) {
                        const int32_t* id = lane_of(q) + g * 128;
                        L.insert(L.end(), id, id + (g == sp ? 3 : 4));
                    }
            std::sort(L.begin(), L.end());
            L.erase(std::unique(L.begin(), L.end()), L.end());
            if ((int64_t)L.size() > dev::kStageMax) continue;  // too wide: the whole structure is dropped below
            for (int64_t q = q0; q < q1; ++q)
                if ((hmeta[q] & 7) == 0)
                    for (int g = 0; g < Kq; ++g)
                        for (int cc = 0; cc < 4; ++cc) {
                            // the freed slot, whose weight is zero, repeats the first member
                            const int id = lane_of(q)[g == sp && cc == 3 ? 0 : g * 128 + cc];
                            hlidx[((size_t)g * np + q) * 4 + cc] =
                                (uint16_t)(std::lower_bound(L.begin(), L.end(), id) - L.begin());
                        }
        }
        hsoff.assign((size_t)nt + 1, 0);
        for (int64_t b = 0; b < nt; ++b) {
            stage_max = std::max(stage_max, (int)lists[(size_t)b].size());
            hsoff[(size_t)b + 1] = hsoff[(size_t)b] + (int)lists[(size_t)b].size();
        }
        if (stage_max <= dev::kStageMax && (int64_t)hsoff.back() < (int64_t)1 << 30) {
            hsids.reserve((size_t)hsoff.back() + 8);
            for (const auto& L : lists) hsids.insert(hsids.end(), L.begin(), L.end());
            hsids.resize((size_t)hsoff.back() + 8, 0);  // the L2 prefetch reads whole 16-byte groups
        } else {
            hlidx.clear();
            hsoff.clear();
            stage_max = 0;
        }
    }
    // ---- device buffers
    float4* dW = nullptr;
    c->S.n_ranges = warp_step_ranges((int)n);
    if (rbf) {
        MLBM_TRY(dalloc(c, &c->idx, (size_t)Kq * np));
        MLBM_TRY(dalloc(c, &dW, (size_t)8 * Kq * np));
    } else {
        MLBM_TRY(dalloc(c, &c->rec, n_words / 4));
        MLBM_TRY(dalloc(c, &c->need, (size_t)np / 32));
        MLBM_TRY(dalloc(c, &c->range, (size_t)c->S.n_ranges + 1));
    }
    MLBM_TRY(dalloc(c, &c->meta, np));
    MLBM_TRY(dalloc(c, &c->mask, np));
    MLBM_TRY(dalloc(c, &c->lag_r, np));
    MLBM_TRY(dalloc(c, &c->link_slot, np));
    MLBM_TRY(dalloc(c, &c->links, hlinks.size()));
    MLBM_TRY(dalloc(c, &c->link_nodes, hlinknodes.size()));
    MLBM_TRY(dalloc(c, &c->eqv, np));
    MLBM_TRY(dalloc(c, &c->perm, np));
    MLBM_TRY(dalloc(c, &c->area, np));
    MLBM_TRY(dalloc(c, &c->area_over_s2, np));
    for (int b = 0; b < 2; ++b) {
        if (p->model == MLBM_MODEL_BGK) {
            MLBM_TRY(dalloc(c, &c->f8[b], (size_t)2 * nps));
            MLBM_TRY(dalloc(c, &c->f0[b], nps));
        } else {
            MLBM_TRY(dalloc(c, &c->ruv[b], nps));
        }
    }
    MLBM_TRY(dalloc(c, &c->rho, np));
    MLBM_TRY(dalloc(c, &c->px, np));
    MLBM_TRY(dalloc(c, &c->py, np));
    MLBM_TRY(dalloc(c, &c->io, (size_t)9 * np));
    if (c->seg_off.empty()) {
        c->seg_off = {0, n};
        c->seg_params = {*p};
        c->seg_box_area = {H.box_area};
    }
    const size_t ns = c->seg_off.size() - 1;
    for (size_t i = 0; i < ns; ++i)
        c->max_blocks = std::max(c->max_blocks, reduce_blocks(c->seg_off[i + 1] - c->seg_off[i]));
    c->link_off.resize(ns + 1);
    for (size_t i = 0; i <= ns; ++i)
        c->link_off[i] = (int)(std::lower_bound(hlinknodes.begin(), hlinknodes.end(), (int)c->seg_off[i]) -
                               hlinknodes.begin());
    c->scratch_len = std::max<int64_t>((int64_t)kObserveBoth * (int64_t)ns * c->max_blocks,
                                       2 * force_blocks(c->n_link_nodes));
    MLBM_TRY(dalloc(c, &c->scratch, c->scratch_len));
    double* results = nullptr;
    MLBM_TRY(dalloc(c, &results, 1 + kObserveBoth * ns));
    c->err = reinterpret_cast<int*>(results);
    c->seg_out = results + 1;
    MLBM_TRY(dalloc(c, &c->seg_dev, ns + 1));
    MLBM_TRY(upload(c, c->seg_dev, c->seg_off.data(), (ns + 1) * sizeof(int64_t)));
    MLBM_CUDA(cudaMemsetAsync(c->err, 0, sizeof(double), c->stream));
    if (!rbf && c->n_halo == 0 && p->model == MLBM_MODEL_BGK) c->cluster = step_cluster_size(Kq, (int)n);
    if (!tma_supported(Kq)) c->variant = 1;  // variants >= 4 exist for K in {12, 16, 24, 32}
    if (rbf) {
        MLBM_TRY(upload(c, c->idx, hidx.data(), hidx.size() * 4));
        MLBM_TRY(upload(c, dW, hW.data(), hW.size() * 4));
    } else {
        MLBM_TRY(upload(c, c->rec, hrec.get(), n_words * 4));
    }
    MLBM_TRY(upload(c, c->meta, hmeta.data(), np));
    MLBM_TRY(upload(c, c->mask, hmask.data(), np));
    MLBM_TRY(upload(c, c->lag_r, hlag.data(), np * 4));
    MLBM_TRY(upload(c, c->link_slot, hslot.data(), np * 4));
    if (!hlinks.empty()) MLBM_TRY(upload(c, c->links, hlinks.data(), hlinks.size() * sizeof(dev::LinkRec)));
    if (!hlinknodes.empty()) MLBM_TRY(upload(c, c->link_nodes, hlinknodes.data(), hlinknodes.size() * 4));
    MLBM_TRY(upload(c, c->eqv, heqv.data(), np * sizeof(float4)));
    MLBM_TRY(upload(c, c->perm, hperm.data(), np * 4));
    MLBM_TRY(upload(c, c->area, harea.data(), np * 4));
    MLBM_TRY(upload(c, c->area_over_s2, has2.data(), np * 4));
    MLBM_CUDA(cudaMemsetAsync(c->px, 0, np * 4, c->stream));
    MLBM_CUDA(cudaMemsetAsync(c->py, 0, np * 4, c->stream));
    for (int b = 0; b < 2; ++b) {
        if (c->f8[b]) {
            MLBM_CUDA(cudaMemsetAsync(c->f8[b], 0, (size_t)2 * nps * sizeof(float4), c->stream));
            MLBM_CUDA(cudaMemsetAsync(c->f0[b], 0, nps * 4, c->stream));
        }
        if (c->ruv[b]) MLBM_CUDA(cudaMemsetAsync(c->ruv[b], 0, nps * sizeof(float4), c->stream));
    }
    c->S.n = (int)n;
    c->S.n_pad = (int)np;
    c->S.K = K;
    c->S.Kq = Kq;
    c->S.bb_mode = H.bb_mode;
    c->S.idx = c->idx;
    c->S.rec = c->rec;
    c->S.need = c->need;
    c->S.range = c->range;
    c->S.rows = rows;
    c->S.meta = c->meta;
    c->S.lag_r = c->lag_r;
    c->S.link_slot = c->link_slot;
    c->S.links = c->links;
    c->S.eqv = c->eqv;
    c->S.link_nodes = c->link_nodes;
    c->S.Wr = dW;
    c->S.n_link_nodes = c->n_link_nodes;
    c->S.lidx = nullptr;
    c->S.stage_off = nullptr;
    c->S.stage_ids = nullptr;
    c->S.stage_max = 0;
    if (!hsoff.empty()) {  // built (a context without least-squares nodes stages nothing)
        ushort4* dl = nullptr;
        int *doff = nullptr, *dids = nullptr;
        MLBM_TRY(dalloc(c, &dl, (size_t)Kq * np));
        MLBM_TRY(dalloc(c, &doff, hsoff.size()));
        MLBM_TRY(dalloc(c, &dids, hsids.size()));
        MLBM_TRY(upload(c, dl, hlidx.data(), hlidx.size() * 2));
        MLBM_TRY(upload(c, doff, hsoff.data(), hsoff.size() * 4));
        MLBM_TRY(upload(c, dids, hsids.data(), hsids.size() * 4));
        if (stage_max > 0) MLBM_CUDA(prepare_staged_step(Kq, stage_max));
        c->S.lidx = dl;
        c->S.stage_off = doff;
        c->S.stage_ids = dids;
        c->S.stage_max = stage_max;
    }
    MLBM_CUDA(launch_record_kinds(c->S, c->rec, c->need, c->range, c->stream));
    if (rbf && p->model == MLBM_MODEL_BGK && (size_t)n * 36 * K > kRbfTilesFrom) {
        MLBM_TRY(build_rbf_tiles(c, false));
        c->rbf_tiles_default = c->S.rbf_rec != nullptr;
    }
    set_collide(c);
    // ---- initial state
    std::vector<double> ru((size_t)n * 3);
    for (int64_t i = 0; i < n; ++i) {
        ru[i * 3] = rho0 ? rho0[i] : 1.0;
        ru[i * 3 + 1] = u0 ? u0[2 * i] : 0.0;
        ru[i * 3 + 2] = u0 ? u0[2 * i + 1] : 0.0;
    }
    MLBM_TRY(upload(c, c->io, ru.data(), ru.size() * 8));
    if (p->model == MLBM_MODEL_BGK) {
        MLBM_CUDA(launch_set_bgk_equilibrium((int)n, c->perm, c->io, c->f8[0], c->f0[0], c->stream));
    } else {
        MLBM_CUDA(launch_set_tau1((int)n, c->perm, c->io, c->ruv[0], c->stream));
    }
    MLBM_CUDA(cudaEventCreate(&c->ev0));
    MLBM_CUDA(cudaEventCreate(&c->ev1));
    return sync(c);
}

// instantiate the graph of kGraphSteps step launches that starts from buffer
// `parity` (capture only: nothing runs, and the state is left as it was)
mlbm_status ensure_graph(mlbm_ctx* c, int parity) {
    cudaGraphExec_t& ex = c->graph[parity];
    if (ex) return MLBM_OK;
    const int saved = c->cur, saved_withhold = c->withhold_next;
    c->cur = parity;
    c->withhold_next = 0;  // never captured into a graph
    cudaGraph_t g = nullptr;
    cudaError_t ee = cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal);
    if (ee != cudaSuccess) {
        c->cur = saved;
        c->withhold_next = saved_withhold;
        return set_error(MLBM_E_CUDA, std::string("graph capture: ") + cudaGetErrorString(ee));
    }
    mlbm_status cs = MLBM_OK;
    for (int i = 0; i < kGraphSteps && cs == MLBM_OK; ++i) cs = launch_one_step(c, c->variant);
    ee = cudaStreamEndCapture(c->stream, &g);
    c->cur = saved;  // an even number of launches returns to it as well
    c->withhold_next = saved_withhold;
    if (cs != MLBM_OK) {
        if (g) cudaGraphDestroy(g);
        return cs;
    }
    if (ee != cudaSuccess) return set_error(MLBM_E_CUDA, std::string("graph capture: ") + cudaGetErrorString(ee));
    ee = cudaGraphInstantiate(&ex, g, 0);
    cudaGraphDestroy(g);
    if (ee != cudaSuccess) {
        ex = nullptr;
        return set_error(MLBM_E_CUDA, std::string("graph instantiate: ") + cudaGetErrorString(ee));
    }
    return MLBM_OK;
}

// graphs are tied to the variant and stream they were captured with
void refresh_graphs(mlbm_ctx* c);

void drop_graphs(mlbm_ctx* c) {
    for (int i = 0; i < 2; ++i)
        if (c->graph[i]) {
            cudaGraphExecDestroy(c->graph[i]);
            c->graph[i] = nullptr;
        }
    c->graph_variant = -1;
}

void refresh_graphs(mlbm_ctx* c) {
    if (c->graph_variant != c->variant || c->graph_stream != c->stream) {
        drop_graphs(c);
        c->graph_variant = c->variant;
        c->graph_stream = c->stream;
    }
}

void free_ctx(mlbm_ctx* c) {
    if (!c) return;
    if (c->stream) cudaStreamSynchronize(c->stream);
    drop_graphs(c);
    for (void* p : c->allocations) cudaFree(p);
    if (c->wall_buf) cudaFree(c->wall_buf);
    if (c->ev0) cudaEventDestroy(c->ev0);
    if (c->ev1) cudaEventDestroy(c->ev1);
    if (c->own_stream) cudaStreamDestroy(c->own_stream);
    delete c;
}

// (rho, u) of every node in the caller's order into FP64 device memory: rows
// [n][3], or (split) rho[n] followed by u[n][2]
mlbm_status fields_to(mlbm_ctx* c, double* out, int split) {
    MLBM_CUDA(launch_macroscopics(c->params.model, (int)c->n, c->perm, c->f8[c->cur], c->f0[c->cur], c->ruv[c->cur],
                                  (float)c->params.gx, (float)c->params.gy, c->S.node_sample, c->S.coll, split, out,
                                  c->stream));
    return MLBM_OK;
}

// observables of every sample into seg_out (see launch_observe)
mlbm_status observe(mlbm_ctx* c, int what, float* px, float* py) {
    dev::Collide C{};  // body force of a single sample as the fields use it
    C.ax = (float)c->params.gx;
    C.ay = (float)c->params.gy;
    MLBM_CUDA(launch_observe(c->params.model, what, (int)c->seg_off.size() - 1, c->max_blocks, c->seg_dev,
                             c->f8[c->cur], c->f0[c->cur], c->ruv[c->cur], C, c->S.coll, c->area, c->mask, px, py,
                             c->scratch, c->seg_out, c->stream));
    return MLBM_OK;
}

// the six field sums over all nodes of a context, as one sample
mlbm_status sums_of_all(mlbm_ctx* c, double* h) {
    if (c->seg_off.size() == 2) {
        MLBM_TRY(observe(c, kObserveFields, nullptr, nullptr));
        return read_results(c, h, 6);
    }
    const size_t ns = c->seg_off.size() - 1;
    std::vector<double> v(6 * ns);
    MLBM_TRY(observe(c, kObserveFields, nullptr, nullptr));
    MLBM_TRY(read_results(c, v.data(), v.size()));
    std::fill(h, h + 6, 0.0);
    for (size_t i = 0; i < ns; ++i)
        for (int q = 0; q < 6; ++q) h[q] += v[6 * i + q];
    return MLBM_OK;
}

// Steady-state iteration shared by the single and batched entry points.
//
// Criterion kFieldNorm (the build's own): every `check` steps each sample's
// velocity is compared with its own snapshot of `window` steps earlier (a
// ring of window / check snapshots), delta = |u(t) - u(t - window)|_2 /
// (window |u(t)|_2) over non-equilibrium nodes; a sample is steady at the
// first t >= window with delta < tol.
//
// Criterion kMeanVelocity (Sec. 3.2): every `check` steps the superficial
// mean velocity <u>(t) = sum u_x A / box area of each sample is recorded; at
// t >= window (the paper's Delta n_t) the relative rate
//   Delta u = |<u>(t) - <u>(t - window)| / (|<u>(t - window)| dt window)
// is formed with the sample's physical time step dt, and the sample is
// steady at the first such t with Delta u < tol (the paper's threshold is
// 1e-2 with Delta n_t = 2e4).  A zero earlier mean is never steady.
//
// Both criteria also check, at every snapshot, that each sample's density is
// positive and its fields finite on every fluid node (MLBM_E_DIVERGED
// otherwise).  at[i] receives the step of sample i's steady state, or -1.
// Steps stop once every sample is steady.  In a tau = 1 batch a sample that
// is steady is held at that state while the others go on (its nodes become
// equilibrium-kind nodes whose record is their state, so each step copies
// it: ~33 B per node update instead of ~473), and it ends at its own steady
// step as a single-sample run does; the kind bytes and records are restored
// when the run ends.
enum SteadyMode { kFieldNorm = 0, kMeanVelocity = 1 };

mlbm_status run_steady(mlbm_ctx* c, int mode, double tol, int64_t window, int64_t check, int64_t max_steps,
                       const double* dt, int64_t* at, const char* name) {
    const std::string nm(name);
    if (!(tol > 0) || window < 1 || check < 1 || window % check != 0 || max_steps < 0)
        return set_error(MLBM_E_INVALID, nm + ": bad arguments (window must be a positive multiple of check)");
    const int ns = (int)c->seg_off.size() - 1;
    if (mode == kMeanVelocity && dt)
        for (int i = 0; i < ns; ++i)
            if (!(dt[i] > 0) || !std::isfinite(dt[i]))
                return set_error(MLBM_E_INVALID, nm + ": time steps must be positive and finite");
    const int64_t R = mode == kFieldNorm ? window / check : 1;
    const int64_t n = c->n;
    std::vector<int64_t> done_at(ns, -1);
    c->steps_in_last_run = 0;
    float* ring = nullptr;
    if (R > 1) {
        if ((double)R * 2.0 * (double)n * 4.0 > 64e9)
            return set_error(MLBM_E_INVALID, nm + ": snapshot ring over 64 GB (use a larger check interval)");
        MLBM_CUDA(cudaMallocAsync(&ring, (size_t)R * 2 * (size_t)n * sizeof(float), c->stream));
    }
    // converged samples of a tau = 1 batch are held (see above)
    uint8_t* saved_meta = nullptr;
    float4* saved_eqv = nullptr;
    bool frozen_any = false;
    if (c->params.model == MLBM_MODEL_TAU1 && ns > 1 && n > 0) {
        const size_t np = (size_t)c->n_pad;
        if (cudaMallocAsync(&saved_meta, np, c->stream) != cudaSuccess ||
            cudaMallocAsync(&saved_eqv, np * sizeof(float4), c->stream) != cudaSuccess) {
            (void)cudaGetLastError();  // no room: every sample steps to the end
            if (saved_meta) cudaFreeAsync(saved_meta, c->stream);
            saved_meta = nullptr;
            saved_eqv = nullptr;
        } else if (cudaMemcpyAsync(saved_meta, c->meta, np, cudaMemcpyDeviceToDevice, c->stream) != cudaSuccess ||
                   cudaMemcpyAsync(saved_eqv, c->eqv, np * sizeof(float4), cudaMemcpyDeviceToDevice,
                                   c->stream) != cudaSuccess) {
            (void)cudaGetLastError();  // nothing frozen yet: step every sample to the end
            cudaFreeAsync(saved_meta, c->stream);
            cudaFreeAsync(saved_eqv, c->stream);
            saved_meta = nullptr;
            saved_eqv = nullptr;
        }
    }
    auto slot_u = [&](int64_t k) { return R > 1 ? ring + (size_t)k * 2 * n : c->px; };
    auto slot_v = [&](int64_t k) { return R > 1 ? ring + ((size_t)k * 2 + 1) * n : c->py; };
    const int what = mode == kMeanVelocity ? kObserveBoth : kObserveChange;
    std::vector<double> h((size_t)what * ns);  // per sample: change sums, then (mean velocity) the field sums
    std::vector<std::vector<double>> hist(ns);  // <u> every `check` steps (mean-velocity criterion)
    // physical time step of each sample: the caller's, else the paper's
    // units (side length 1, kinematic viscosity 1): dt = nu_lb (s / L)^2 with
    // L the side of a square of the sample's box area
    std::vector<double> dts(ns, 1.0);
    for (int i = 0; i < ns; ++i) {
        const double si = c->seg_s.empty() ? c->s : c->seg_s[i];
        const double L = std::sqrt(c->seg_box_area[i]);
        dts[i] = dt ? dt[i] : (c->seg_params[i].tau - 0.5) / 3.0 * (si / L) * (si / L);
    }
    auto snapshot = [&](int64_t k) -> mlbm_status {
        MLBM_TRY(observe(c, what, slot_u(k), slot_v(k)));
        MLBM_TRY(read_results(c, h.data(), h.size()));
        for (int i = 0; i < ns; ++i) {
            const double* v = &h[(size_t)what * i];
            if (v[2] != 0.0 || !std::isfinite(v[0]) || !std::isfinite(v[1]))
                return set_error(MLBM_E_DIVERGED, nm + ": non-positive density or non-finite field in sample " +
                                                      std::to_string(i) + " (" +
                                                      std::to_string((int64_t)v[2]) + " nodes)");
            if (mode == kMeanVelocity) hist[i].push_back(v[5] / c->seg_box_area[i]);
        }
        return MLBM_OK;
    };
    auto body = [&]() -> mlbm_status {
        MLBM_TRY(snapshot(0));
        int64_t t = 0;
        int remaining = ns;
        while (t < max_steps && remaining > 0) {
            const int64_t w = std::min(check, max_steps - t);
            MLBM_TRY(mlbm_step(c, w));
            t += w;
            c->steps_in_last_run = t;
            if (w != check) break;  // a partial chunk at max_steps is not evaluated
            MLBM_TRY(snapshot((t / check) % R));
            if (t < window) continue;
            for (int i = 0; i < ns; ++i) {
                if (done_at[i] >= 0) continue;
                bool steady;
                if (mode == kFieldNorm) {
                    const double* v = &h[(size_t)what * i];
                    const double delta = v[1] > 0 ? std::sqrt(v[0] / v[1]) / (double)window : 0.0;
                    steady = delta < tol;
                } else {
                    const size_t j = hist[i].size() - 1, lag = (size_t)(window / check);
                    const double now = hist[i][j], then = hist[i][j - lag];
                    steady = then != 0.0 && std::fabs(now - then) / (std::fabs(then) * dts[i] * (double)window) < tol;
                }
                if (steady) {
                    done_at[i] = t;
                    --remaining;
                    if (saved_meta && remaining > 0) {
                        const int64_t o = c->seg_off[i];
                        MLBM_CUDA(launch_freeze_tau1((int)o, (int)(c->seg_off[i + 1] - o), c->meta, c->eqv,
                                                     c->ruv[c->cur], c->stream));
                        MLBM_CUDA(launch_record_kinds(c->S, c->rec, c->need, c->range, c->stream));
                        MLBM_TRY(sync(c));
                        frozen_any = true;
                    }
                }
            }
        }
        return remaining == 0 ? MLBM_OK : set_error(MLBM_E_NOT_CONVERGED, nm + ": max_steps reached");
    };
    mlbm_status st = body();
    if (frozen_any) {
        const size_t np = (size_t)c->n_pad;
        cudaMemcpyAsync(c->meta, saved_meta, np, cudaMemcpyDeviceToDevice, c->stream);
        cudaMemcpyAsync(c->eqv, saved_eqv, np * sizeof(float4), cudaMemcpyDeviceToDevice, c->stream);
        launch_record_kinds(c->S, c->rec, c->need, c->range, c->stream);
    }
    if (saved_meta) cudaFreeAsync(saved_meta, c->stream);
    if (saved_eqv) cudaFreeAsync(saved_eqv, c->stream);
    if (ring) cudaFreeAsync(ring, c->stream);
    if (ring || saved_meta) cudaStreamSynchronize(c->stream);  // also before the next step reads the kinds
    if (at)
        for (int i = 0; i < ns; ++i) at[i] = done_at[i];
    return st;
}

}  // namespace


extern "C" {

const char* mlbm_last_error(void) { return mlbm::g_last_error.c_str(); }

const char* mlbm_version(void) { return "mlbm-gb300 0.1 (sm_103a)"; }

mlbm_status mlbm_init(mlbm_ctx** out, const mlbm_stencils* st, const mlbm_params* p, const double* rho0,
                      const double* u0) {
    clear_error();
    if (!out || !st || !p) return set_error(MLBM_E_INVALID, "init: NULL argument");
    *out = nullptr;
    MLBM_TRY(check_params(p));
    int ndev = 0;
    cudaError_t e = cudaGetDeviceCount(&ndev);
    if (e != cudaSuccess || ndev == 0) {
        (void)cudaGetLastError();
        return set_error(MLBM_E_CUDA, std::string("init: no CUDA device (") + cudaGetErrorString(e) + ")");
    }
    auto* c = new (std::nothrow) mlbm_ctx;
    if (!c) return set_error(MLBM_E_OOM, "init: out of host memory");
    mlbm_status s = do_init(c, st, p, rho0, u0);
    if (s != MLBM_OK) {
        std::string msg = g_last_error;
        free_ctx(c);
        return set_error(s, msg);
    }
    *out = c;
    return MLBM_OK;
}

void mlbm_destroy(mlbm_ctx* ctx) { free_ctx(ctx); }

mlbm_status mlbm_set_stream(mlbm_ctx* c, void* stream) {
    if (!c) return set_error(MLBM_E_INVALID, "set_stream: NULL context");
    MLBM_CUDA(cudaStreamSynchronize(c->stream));
    c->stream = stream ? static_cast<cudaStream_t>(stream) : c->own_stream;
    return MLBM_OK;
}

mlbm_status mlbm_set_populations(mlbm_ctx* c, const double* f) {
    if (!c || !f) return set_error(MLBM_E_INVALID, "set_populations: NULL argument");
    if (c->params.model != MLBM_MODEL_BGK) return set_error(MLBM_E_INVALID, "set_populations: BGK contexts only");
    MLBM_TRY(upload(c, c->io, f, (size_t)c->n * 9 * 8));
    MLBM_CUDA(launch_set_bgk((int)c->n, c->perm, c->io, c->f8[c->cur], c->f0[c->cur], c->stream));
    c->steps = 0;
    return sync(c);
}

mlbm_status mlbm_set_fields(mlbm_ctx* c, const double* ru) {
    if (!c || !ru) return set_error(MLBM_E_INVALID, "set_fields: NULL argument");
    MLBM_TRY(upload(c, c->io, ru, (size_t)c->n * 3 * 8));
    if (c->params.model == MLBM_MODEL_BGK)
        MLBM_CUDA(launch_set_bgk_equilibrium((int)c->n, c->perm, c->io, c->f8[c->cur], c->f0[c->cur], c->stream));
    else
        MLBM_CUDA(launch_set_tau1((int)c->n, c->perm, c->io, c->ruv[c->cur], c->stream));
    c->steps = 0;
    return sync(c);
}

mlbm_status mlbm_get_populations(mlbm_ctx* c, double* f) {
    if (!c || !f) return set_error(MLBM_E_INVALID, "get_populations: NULL argument");
    if (c->params.model != MLBM_MODEL_BGK) return set_error(MLBM_E_INVALID, "get_populations: BGK contexts only");
    MLBM_CUDA(launch_get_bgk((int)c->n, c->perm, c->f8[c->cur], c->f0[c->cur], c->io, c->stream));
    MLBM_CUDA(cudaMemcpyAsync(f, c->io, (size_t)c->n * 9 * 8, cudaMemcpyDeviceToHost, c->stream));
    return sync(c);
}

mlbm_status mlbm_get_fields(mlbm_ctx* c, double* ru) {
    if (!c || !ru) return set_error(MLBM_E_INVALID, "get_fields: NULL argument");
    MLBM_TRY(fields_to(c, c->io, 0));
    MLBM_CUDA(cudaMemcpyAsync(ru, c->io, (size_t)c->n * 3 * 8, cudaMemcpyDeviceToHost, c->stream));
    return sync(c);
}

mlbm_status mlbm_step(mlbm_ctx* c, int64_t n_steps) {
    if (!c) return set_error(MLBM_E_INVALID, "step: NULL context");
    if (n_steps < 0) return set_error(MLBM_E_INVALID, "step: negative step count");
    if (n_steps == 0) return MLBM_OK;
    if (c->timing) MLBM_CUDA(cudaEventRecord(c->ev0, c->stream));
    int64_t left = n_steps;
    if (by_cluster(c, n_steps, c->variant)) {
        MLBM_TRY(launch_cluster_steps(c, n_steps));
        left = 0;
    }
    // a launch that must withhold a tile runs directly, not from a graph
    else if (c->use_graphs && n_steps >= kGraphSteps && !c->withhold_next) {
        refresh_graphs(c);
        while (left >= kGraphSteps) {
            MLBM_TRY(ensure_graph(c, c->cur));
            MLBM_CUDA(cudaGraphLaunch(c->graph[c->cur], c->stream));
            left -= kGraphSteps;
        }
    }
    for (int64_t t = 0; t < left; ++t) MLBM_TRY(launch_one_step(c, c->variant));
    c->steps += n_steps;
    if (c->timing) {
        MLBM_CUDA(cudaEventRecord(c->ev1, c->stream));
        MLBM_CUDA(cudaEventSynchronize(c->ev1));
        float ms = 0.f;
        MLBM_CUDA(cudaEventElapsedTime(&ms, c->ev0, c->ev1));
        c->last_ms = ms / (double)n_steps;
    }
    return MLBM_OK;
}

mlbm_status mlbm_prepare_graphs(mlbm_ctx* c) {
    if (!c) return set_error(MLBM_E_INVALID, "prepare_graphs: NULL context");
    if (!c->use_graphs || by_cluster(c, kGraphSteps, c->variant)) return MLBM_OK;
    refresh_graphs(c);
    MLBM_TRY(ensure_graph(c, 0));
    MLBM_TRY(ensure_graph(c, 1));
    return MLBM_OK;
}

mlbm_status mlbm_set_wait_limit(mlbm_ctx* c, double seconds) {
    if (!c) return set_error(MLBM_E_INVALID, "set_wait_limit: NULL context");
    if (!(seconds >= 1e-4 && seconds <= 60.0))
        return set_error(MLBM_E_INVALID, "set_wait_limit: the limit must lie in [1e-4, 60] seconds");
    c->wait_ns = (unsigned long long)(seconds * 1e9);
    drop_graphs(c);  // captured launches carry the old limit
    return MLBM_OK;
}

mlbm_status mlbm_test_withhold_copy(mlbm_ctx* c) {
    if (!c) return set_error(MLBM_E_INVALID, "test_withhold_copy: NULL context");
    if (!((c->variant >= 4 && c->variant <= 7) || (c->variant >= 27 && c->variant <= 29)) || c->S.Wr)
        return set_error(MLBM_E_INVALID, "test_withhold_copy: the context's kernel variant has no bulk-copy ring");
    c->withhold_next = 1;
    return MLBM_OK;
}

int64_t mlbm_step_count(const mlbm_ctx* c) { return c ? c->steps : -1; }

mlbm_status mlbm_set_timing(mlbm_ctx* c, int enable) {
    if (!c) return set_error(MLBM_E_INVALID, "set_timing: NULL context");
    c->timing = enable != 0;
    c->last_ms = -1.0;
    return MLBM_OK;
}

double mlbm_last_step_ms(const mlbm_ctx* c) { return c ? c->last_ms : -1.0; }

mlbm_status mlbm_macroscopics(mlbm_ctx* c, double* rho, double* u) {
    if (!c) return set_error(MLBM_E_INVALID, "macroscopics: NULL context");
    if (!rho && !u) return sync(c);
    MLBM_TRY(fields_to(c, c->io, 1));
    const size_t n = (size_t)c->n;
    if (rho) MLBM_CUDA(cudaMemcpyAsync(rho, c->io, n * 8, cudaMemcpyDeviceToHost, c->stream));
    if (u) MLBM_CUDA(cudaMemcpyAsync(u, c->io + n, n * 16, cudaMemcpyDeviceToHost, c->stream));
    return sync(c);
}

mlbm_status mlbm_wall_stress_force(mlbm_ctx* c, const int64_t* nodes, const double* normals, const double* ds,
                                   int64_t m, double* fx, double* fy) {
    if (!c || (m > 0 && (!nodes || !normals || !ds)) || m < 0)
        return set_error(MLBM_E_INVALID, "wall_stress_force: bad arguments");
    if (c->seg_off.size() > 2) return set_error(MLBM_E_INVALID, "wall_stress_force: single-sample contexts only");
    if (c->S.Wr) return set_error(MLBM_E_INVALID, "wall_stress_force: least-squares stencils only");
    if (m > (int64_t)1 << 30) return set_error(MLBM_E_INVALID, "wall_stress_force: too many wall nodes");
    // caller's node ids -> device positions
    std::vector<int> pos((size_t)m);
    for (int64_t i = 0; i < m; ++i) {
        if (nodes[i] < 0 || nodes[i] >= c->n) return set_error(MLBM_E_INVALID, "wall_stress_force: node id out of range");
        pos[(size_t)i] = c->inv_perm[(size_t)nodes[i]];
    }
    double sx = 0.0, sy = 0.0;
    if (m > 0) {
        const size_t mm = (size_t)m;
        if (m > c->wall_cap) {  // grow (rare: the wall node list is usually fixed)
            if (c->wall_buf) {
                MLBM_CUDA(cudaStreamSynchronize(c->stream));
                cudaFree(c->wall_buf);
                c->wall_buf = nullptr;
                c->wall_cap = 0;
            }
            void* q = nullptr;
            cudaError_t e = cudaMalloc(&q, mm * 48);
            if (e != cudaSuccess) {
                (void)cudaGetLastError();
                return set_error(MLBM_E_OOM, std::string("wall_stress_force: cudaMalloc: ") + cudaGetErrorString(e));
            }
            c->wall_buf = static_cast<uint8_t*>(q);
            c->wall_cap = m;
        }
        // normals | tractions | lengths | positions (16-, 16-, 8-, 4-byte items)
        const size_t cap = (size_t)c->wall_cap;
        double* dn = reinterpret_cast<double*>(c->wall_buf);
        double* dout = reinterpret_cast<double*>(c->wall_buf + cap * 16);
        double* dds = reinterpret_cast<double*>(c->wall_buf + cap * 32);
        int* dpos = reinterpret_cast<int*>(c->wall_buf + cap * 40);
        std::vector<double> out(2 * mm, 0.0);
        cudaError_t e = cudaMemcpyAsync(dpos, pos.data(), mm * 4, cudaMemcpyHostToDevice, c->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(dn, normals, mm * 16, cudaMemcpyHostToDevice, c->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(dds, ds, mm * 8, cudaMemcpyHostToDevice, c->stream);
        if (e == cudaSuccess) {
            const int model = c->params.model == MLBM_MODEL_BGK ? 0 : 1;
            const double nu = (c->params.tau - 0.5) / 3.0;
            e = launch_wall_traction(c->S, model, c->f8[c->cur], c->f0[c->cur], c->ruv[c->cur], c->C.ax, c->C.ay,
                                     nu, c->s, dpos, dn, dds, (int)m, dout, c->stream);
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(out.data(), dout, mm * 16, cudaMemcpyDeviceToHost, c->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
        if (e != cudaSuccess) return set_error(MLBM_E_CUDA, std::string("wall_stress_force: ") + cudaGetErrorString(e));
        for (size_t i = 0; i < mm; ++i) {  // fixed order: reproducible
            if (std::isnan(out[2 * i])) return set_error(MLBM_E_INVALID, "wall_stress_force: node " +
                                                                         std::to_string(nodes[i]) +
                                                                         " is not a least-squares node");
            sx += out[2 * i];
            sy += out[2 * i + 1];
        }
    }
    if (fx) *fx = sx;
    if (fy) *fy = sy;
    return MLBM_OK;
}

mlbm_status mlbm_drag_lift(mlbm_ctx* c, double ref_length, double u_ref, double* fx, double* fy, double* cd,
                           double* cl) {
    if (!c) return set_error(MLBM_E_INVALID, "drag_lift: NULL context");
    double h[2] = {0, 0};
    if (c->n_link_nodes > 0) {
        MLBM_CUDA(launch_force(c->S, c->params.model, c->n_link_nodes, c->link_nodes, c->area_over_s2,
                               c->f8[c->cur], c->ruv[c->cur], c->C, c->scratch, c->seg_out, c->stream));
        MLBM_TRY(read_results(c, h, 2));
    }
    if (fx) *fx = h[0];
    if (fy) *fy = h[1];
    const double L = ref_length / c->s;
    const double den = u_ref * u_ref * L;
    if (cd) *cd = den != 0 ? 2.0 * h[0] / den : 0.0;
    if (cl) *cl = den != 0 ? 2.0 * h[1] / den : 0.0;
    return MLBM_OK;
}

mlbm_status mlbm_permeability(mlbm_ctx* c, double* k, double* us, double* ui, double* tort) {
    if (!c) return set_error(MLBM_E_INVALID, "permeability: NULL context");
    double h[6];
    MLBM_TRY(sums_of_all(c, h));
    const double sup = h[2] / c->box_area;
    const double gmag = std::sqrt(c->params.gx * c->params.gx + c->params.gy * c->params.gy);
    const double nu = (c->params.tau - 0.5) / 3.0;
    if (us) *us = sup;
    if (ui) *ui = h[0] != 0 ? h[2] / h[0] : 0.0;
    if (k) *k = gmag > 0 ? nu * sup / gmag : 0.0;
    if (tort) *tort = h[2] != 0 ? h[4] / h[2] : 0.0;
    return MLBM_OK;
}

mlbm_status mlbm_run_to_steady(mlbm_ctx* c, double tol, int64_t window, int64_t max_steps, int64_t* taken) {
    return mlbm_run_to_steady_ex(c, tol, window, window, max_steps, taken);
}

mlbm_status mlbm_run_to_steady_ex(mlbm_ctx* c, double tol, int64_t window, int64_t check, int64_t max_steps,
                                  int64_t* taken) {
    if (!c) return set_error(MLBM_E_INVALID, "run_to_steady: NULL context");
    if (taken) *taken = 0;
    int64_t at = -1;
    mlbm_status st = run_steady(c, kFieldNorm, tol, window, check, max_steps, nullptr, &at, "run_to_steady");
    if (taken) *taken = at >= 0 ? at : c->steps_in_last_run;
    return st;
}

mlbm_status mlbm_run_to_steady_mean(mlbm_ctx* c, double threshold, int64_t dn, int64_t check, double dt,
                                    int64_t max_steps, int64_t* taken) {
    if (!c) return set_error(MLBM_E_INVALID, "run_to_steady_mean: NULL context");
    if (taken) *taken = 0;
    if (c->seg_off.size() != 2) return set_error(MLBM_E_INVALID, "run_to_steady_mean: batched context");
    int64_t at = -1;
    const double* dtp = dt > 0 ? &dt : nullptr;
    if (dt < 0 || !std::isfinite(dt)) return set_error(MLBM_E_INVALID, "run_to_steady_mean: bad time step");
    mlbm_status st = run_steady(c, kMeanVelocity, threshold, dn, check, max_steps, dtp, &at, "run_to_steady_mean");
    if (taken) *taken = at >= 0 ? at : c->steps_in_last_run;
    return st;
}

mlbm_status mlbm_save(mlbm_ctx* c, const char* path) {
    if (!c || !path) return set_error(MLBM_E_INVALID, "save: NULL argument");
    const int per = c->params.model == MLBM_MODEL_BGK ? 9 : 3;
    std::vector<double> buf((size_t)c->n * per);
    MLBM_TRY(per == 9 ? mlbm_get_populations(c, buf.data()) : mlbm_get_fields(c, buf.data()));
    FILE* f = std::fopen(path, "wb");
    if (!f) return set_error(MLBM_E_IO, std::string("save: cannot open ") + path);
    const char magic[8] = {'M', 'L', 'B', 'M', 'S', 'T', '0', '1'};
    int64_t hdr[4] = {c->n, c->K, c->params.model, c->steps};
    bool ok = std::fwrite(magic, 1, 8, f) == 8 && std::fwrite(hdr, 8, 4, f) == 4 &&
              std::fwrite(&c->params, sizeof(mlbm_params), 1, f) == 1 &&
              std::fwrite(buf.data(), 8, buf.size(), f) == buf.size();
    ok = (std::fclose(f) == 0) && ok;
    return ok ? MLBM_OK : set_error(MLBM_E_IO, "save: write failed");
}

mlbm_status mlbm_load(mlbm_ctx* c, const char* path) {
    if (!c || !path) return set_error(MLBM_E_INVALID, "load: NULL argument");
    FILE* f = std::fopen(path, "rb");
    if (!f) return set_error(MLBM_E_IO, std::string("load: cannot open ") + path);
    char magic[8];
    int64_t hdr[4];
    mlbm_params p;
    bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, "MLBMST01", 8) == 0 &&
              std::fread(hdr, 8, 4, f) == 4 && std::fread(&p, sizeof(p), 1, f) == 1;
    if (!ok || hdr[0] != c->n || hdr[1] != c->K || hdr[2] != c->params.model) {
        std::fclose(f);
        return set_error(MLBM_E_IO, "load: file does not match this context");
    }
    const int per = c->params.model == MLBM_MODEL_BGK ? 9 : 3;
    std::vector<double> buf((size_t)c->n * per);
    ok = std::fread(buf.data(), 8, buf.size(), f) == buf.size();
    std::fclose(f);
    if (!ok) return set_error(MLBM_E_IO, "load: truncated file");
    // every copy of a single sample's parameters: the host's, those in captured
    // steps, and the table of a batch of one (a larger batch keeps its samples'
    // own, which the file does not hold)
    MLBM_CUDA(cudaStreamSynchronize(c->stream));
    drop_graphs(c);
    c->params = p;
    set_collide(c);
    if (c->seg_params.size() == 1) {
        c->seg_params[0] = p;
        if (c->S.coll)
            MLBM_TRY(upload(c, const_cast<dev::Collide*>(c->S.coll), &c->C, sizeof(dev::Collide)));
    }
    if (per == 9) {
        MLBM_TRY(upload(c, c->io, buf.data(), buf.size() * 8));
        MLBM_CUDA(launch_set_bgk((int)c->n, c->perm, c->io, c->f8[c->cur], c->f0[c->cur], c->stream));
    } else {
        MLBM_TRY(upload(c, c->io, buf.data(), buf.size() * 8));
        MLBM_CUDA(launch_set_tau1((int)c->n, c->perm, c->io, c->ruv[c->cur], c->stream));
    }
    MLBM_TRY(sync(c));
    c->steps = hdr[3];
    return MLBM_OK;
}

mlbm_status mlbm_set_kernel_variant(mlbm_ctx* c, int variant) {
    if (!c) return set_error(MLBM_E_INVALID, "set_kernel_variant: NULL context");
    if (variant < 0 || variant > kMaxVariant || (variant >= 4 && !tma_supported(c->K / 4)))
        return set_error(MLBM_E_INVALID, "set_kernel_variant: variant not available for this K");
    if (variant == 22 && c->params.model == MLBM_MODEL_BGK && !c->S.Wr && !c->S.lidx)
        return set_error(MLBM_E_INVALID, "set_kernel_variant: no staged neighbourhoods for this context");
    if ((variant == 28 || variant == 29) && c->S.Wr && c->params.model == MLBM_MODEL_BGK && !c->S.rbf_rec)
        MLBM_TRY(build_rbf_tiles(c, true));
    c->variant = variant;
    return MLBM_OK;
}

int mlbm_kernel_variant(const mlbm_ctx* c) { return c ? c->variant : -1; }

int mlbm_autotune_times(const mlbm_ctx* c, double* ms, int n) {
    if (!c) return -1;
    for (int v = 0; v < n && v <= kMaxVariant; ++v)
        ms[v] = v < (int)c->tune_ms.size() ? c->tune_ms[v] : -1.0;
    return kMaxVariant + 1;
}

mlbm_status mlbm_autotune(mlbm_ctx* c, int steps_per_variant, double* best_ms) {
    return mlbm_autotune_ex(c, steps_per_variant, 0, best_ms);
}

mlbm_status mlbm_autotune_ex(mlbm_ctx* c, int steps_per_variant, int flush_l2, double* best_ms) {
    if (!c || steps_per_variant < 1) return set_error(MLBM_E_INVALID, "autotune: bad arguments");
    // optional L2 flush between timed steps: a zeroed 512 MiB device buffer
    // read before every step, so each timed step reads its stencil data from
    // HBM and starts with no dirty lines in L2
    void* flush = nullptr;
    const size_t flush_bytes = size_t(512) << 20;
    if (flush_l2 && cudaMalloc(&flush, flush_bytes) != cudaSuccess) {
        (void)cudaGetLastError();
        return set_error(MLBM_E_OOM, "autotune: no room for the L2 flush buffer");
    }
    if (flush_l2 && cudaMemsetAsync(flush, 0, flush_bytes, c->stream) != cudaSuccess) {
        cudaFree(flush);
        return set_error(MLBM_E_CUDA, "autotune: flush buffer memset failed");
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (flush_l2) {
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
    }
    // keep the state: tuning steps run on a copy and the buffers are restored
    const size_t np = (size_t)c->n_pad;
    std::vector<void*> saved;
    auto save_buf = [&](void* d, size_t bytes) -> mlbm_status {
        void* q = nullptr;
        if (cudaMalloc(&q, bytes) != cudaSuccess) {
            (void)cudaGetLastError();
            return set_error(MLBM_E_OOM, "autotune: no room for a state copy");
        }
        saved.push_back(q);
        MLBM_CUDA(cudaMemcpyAsync(q, d, bytes, cudaMemcpyDeviceToDevice, c->stream));
        return MLBM_OK;
    };
    const int cur0 = c->cur;
    const int64_t steps0 = c->steps;
    mlbm_status st = MLBM_OK;
    if (c->params.model == MLBM_MODEL_BGK) {
        st = save_buf(c->f8[cur0], 2 * np * sizeof(float4));
        if (st == MLBM_OK) st = save_buf(c->f0[cur0], np * sizeof(float));
    } else {
        st = save_buf(c->ruv[cur0], np * sizeof(float4));
    }
    // RBF-FD stencils: 28 and 29 step from tile records, as after set_kernel_variant
    const bool had_rbf_tiles = c->S.rbf_rec != nullptr;
    if (st == MLBM_OK && c->S.Wr && c->params.model == MLBM_MODEL_BGK && tma_supported(c->K / 4) && !had_rbf_tiles)
        st = build_rbf_tiles(c, true);
    int best = c->variant;
    double best_t = 1e30;
    c->tune_ms.assign(kMaxVariant + 1, -1.0);
    for (int v = 0; v <= kMaxVariant && st == MLBM_OK; ++v) {
        if (v >= 14 && v <= 24 && c->params.model != MLBM_MODEL_BGK) continue;
        if (v >= 4 && !tma_supported(c->K / 4)) continue;
        // one untimed warm-up launch, then the timed ones
        st = launch_one_step(c, v);
        if (st != MLBM_OK) {  // a variant that cannot launch here (resources) is skipped
            (void)cudaGetLastError();
            st = MLBM_OK;
            continue;
        }
        double per = 0.0;
        if (flush_l2) {
            double tot = 0.0;
            for (int i = 0; i < steps_per_variant && st == MLBM_OK; ++i) {
                l2_flush_read<<<152 * 8, 256, 0, c->stream>>>(static_cast<const float4*>(flush),
                                                               flush_bytes / sizeof(float4),
                                                               static_cast<float*>(flush));
                cudaEventRecord(e0, c->stream);
                st = launch_one_step(c, v);
                cudaEventRecord(e1, c->stream);
                if (cudaEventSynchronize(e1) != cudaSuccess) {
                    st = set_error(MLBM_E_CUDA, "autotune: event wait failed");
                    break;
                }
                float ms = 0.f;
                cudaEventElapsedTime(&ms, e0, e1);
                tot += ms;
            }
            if (st != MLBM_OK) break;
            per = tot / steps_per_variant;
        } else {
            if (cudaEventRecord(c->ev0, c->stream) != cudaSuccess) break;
            if (by_cluster(c, steps_per_variant, v))
                st = launch_cluster_steps(c, steps_per_variant);
            else
                for (int i = 0; i < steps_per_variant && st == MLBM_OK; ++i) st = launch_one_step(c, v);
            if (st != MLBM_OK) break;
            cudaEventRecord(c->ev1, c->stream);
            if (cudaEventSynchronize(c->ev1) != cudaSuccess) {
                st = set_error(MLBM_E_CUDA, "autotune: event wait failed");
                break;
            }
            float ms = 0.f;
            cudaEventElapsedTime(&ms, c->ev0, c->ev1);
            per = ms / steps_per_variant;
        }
        c->tune_ms[v] = per;
        if (per < best_t) {
            best_t = per;
            best = v;
        }
    }
    // restore
    if (st == MLBM_OK) {
        c->cur = cur0;
        if (c->params.model == MLBM_MODEL_BGK) {
            cudaMemcpyAsync(c->f8[cur0], saved[0], 2 * np * sizeof(float4), cudaMemcpyDeviceToDevice, c->stream);
            cudaMemcpyAsync(c->f0[cur0], saved[1], np * sizeof(float), cudaMemcpyDeviceToDevice, c->stream);
        } else {
            cudaMemcpyAsync(c->ruv[cur0], saved[0], np * sizeof(float4), cudaMemcpyDeviceToDevice, c->stream);
        }
        st = sync(c);
    }
    for (void* q : saved) cudaFree(q);
    if (flush) cudaFree(flush);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    c->steps = steps0;
    if (st == MLBM_OK) c->variant = best;
    // records that the chosen number does not step from are given back
    if (!had_rbf_tiles && c->S.rbf_rec && !by_rbf_tiles(c, c->variant)) {
        cudaStreamSynchronize(c->stream);  // and no graph holds them: they were not there before
        drop_rbf_tiles(c);
    }
    if (st != MLBM_OK) return st;
    if (best_ms) *best_ms = best_t;
    return MLBM_OK;
}

mlbm_status mlbm_batch_init(mlbm_ctx** out, const mlbm_stencils* const* sts, const mlbm_params* params,
                            int n_samples) {
    clear_error();
    if (!out || !sts || !params || n_samples < 1 || n_samples > 65535)
        return set_error(MLBM_E_INVALID, "batch_init: bad arguments");
    *out = nullptr;
    for (int i = 0; i < n_samples; ++i) {
        if (!sts[i]) return set_error(MLBM_E_INVALID, "batch_init: NULL stencils");
        MLBM_TRY(check_params(&params[i]));
        if (sts[i]->h.K != sts[0]->h.K || sts[i]->h.bb_mode != sts[0]->h.bb_mode ||
            params[i].model != params[0].model || sts[i]->h.interp != sts[0]->h.interp)
            return set_error(MLBM_E_INVALID,
                             "batch_init: samples must share K, bounce-back rule, interpolant and model");
    }
    // concatenate the samples' host stencils; sample i keeps its own Hilbert
    // order inside positions [off_i, off_i + n_i)
    auto* cat = new (std::nothrow) mlbm_stencils;
    if (!cat) return set_error(MLBM_E_OOM, "batch_init: out of host memory");
    HostStencils& C = cat->h;
    const int K = sts[0]->h.K;
    C.K = K;
    C.s = sts[0]->h.s;
    C.bb_mode = sts[0]->h.bb_mode;
    C.interp = sts[0]->h.interp;
    std::vector<int64_t> off(n_samples + 1, 0);
    for (int i = 0; i < n_samples; ++i) off[i + 1] = off[i] + sts[i]->h.n;
    const int64_t n = off[n_samples];
    if (n > (int64_t(1) << 31) - 1) {
        delete cat;
        return set_error(MLBM_E_INVALID, "batch_init: more than 2^31 - 1 nodes in total");
    }
    C.n = n;
    C.box_area = 0;
    C.perm.resize(n); C.inv.resize(n); C.idx.resize((size_t)n * K);
    C.kind.resize(n); C.center.resize(n); C.lag_h.resize(n); C.lag_slot.resize((size_t)n * 9);
    C.link_mask.resize(n); C.q.resize((size_t)n * 9); C.eqv.resize((size_t)n * 3); C.area.resize(n);
    C.s_node.resize(n);
    std::vector<uint16_t> node_sample(n);
    for (int i = 0; i < n_samples; ++i) {
        const HostStencils& H = sts[i]->h;
        const int64_t o = off[i];
        const bool wr = C.interp != MLBM_INTERP_WLS;
        // the matrix and weight rows stay in the sample's stencils
        C.part_M.push_back(H.M.data());
        C.part_Wr.push_back(wr ? H.Wr.data() : nullptr);
        // every node's rows in parallel (each node writes only its own)
#pragma omp parallel for schedule(static, 4096)
        for (int64_t p = 0; p < H.n; ++p) {
            const size_t g = (size_t)(o + p);
            C.perm[g] = o + H.perm[p];
            C.inv[o + H.perm[p]] = o + p;
            for (int j = 0; j < K; ++j) C.idx[g * K + j] = (int32_t)(o + H.idx[(size_t)p * K + j]);
            std::copy_n(H.lag_slot.begin() + (size_t)p * 9, 9, C.lag_slot.begin() + g * 9);
            std::copy_n(H.q.begin() + (size_t)p * 9, 9, C.q.begin() + g * 9);
            std::copy_n(H.eqv.begin() + (size_t)p * 3, 3, C.eqv.begin() + g * 3);
            C.kind[g] = H.kind[p];
            C.center[g] = H.center[p];
            C.lag_h[g] = H.lag_h[p];
            C.link_mask[g] = H.link_mask[p];
            C.area[g] = H.area[p];
            C.s_node[g] = H.s;
            node_sample[g] = (uint16_t)i;
        }
        C.info.n_wls += H.info.n_wls;
        C.info.n_lagrange += H.info.n_lagrange;
        C.info.n_eq += H.info.n_eq;
        C.info.n_link_nodes += H.info.n_link_nodes;
        C.info.n_links += H.info.n_links;
    }
    C.part_off = off;
    C.info.n = n;
    C.info.K = K;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
        (void)cudaGetLastError();
        delete cat;
        return set_error(MLBM_E_CUDA, "batch_init: no CUDA device");
    }
    auto* c = new (std::nothrow) mlbm_ctx;
    if (!c) {
        delete cat;
        return set_error(MLBM_E_OOM, "batch_init: out of host memory");
    }
    c->seg_off = off;
    c->seg_params.assign(params, params + n_samples);
    for (int i = 0; i < n_samples; ++i) {
        c->seg_box_area.push_back(sts[i]->h.box_area);
        c->seg_s.push_back(sts[i]->h.s);
    }
    mlbm_status st = do_init(c, cat, &params[0], nullptr, nullptr);
    delete cat;
    if (st == MLBM_OK) {
        // per-sample collision table and per-node sample index
        std::vector<dev::Collide> table(n_samples);
        for (int i = 0; i < n_samples; ++i) {
            mlbm_ctx tmp;
            tmp.params = params[i];
            set_collide(&tmp);
            table[i] = tmp.C;
        }
        uint16_t* d_ns = nullptr;
        dev::Collide* d_coll = nullptr;
        st = dalloc(c, &d_ns, (size_t)c->n_pad);
        if (st == MLBM_OK) st = dalloc(c, &d_coll, (size_t)n_samples);
        if (st == MLBM_OK) st = upload(c, d_ns, node_sample.data(), (size_t)n * 2);
        if (st == MLBM_OK) st = upload(c, d_coll, table.data(), table.size() * sizeof(dev::Collide));
        if (st == MLBM_OK) {
            c->S.node_sample = d_ns;
            c->S.coll = d_coll;
            st = sync(c);
        }
    }
    if (st != MLBM_OK) {
        std::string msg = g_last_error;
        free_ctx(c);
        return set_error(st, msg);
    }
    *out = c;
    return MLBM_OK;
}

int mlbm_batch_size(const mlbm_ctx* c) { return c ? (int)c->seg_off.size() - 1 : -1; }

mlbm_status mlbm_batch_range(const mlbm_ctx* c, int sample, int64_t* first, int64_t* count) {
    if (!c || sample < 0 || sample >= (int)c->seg_off.size() - 1) return set_error(MLBM_E_INVALID, "batch_range: bad sample");
    if (first) *first = c->seg_off[sample];
    if (count) *count = c->seg_off[sample + 1] - c->seg_off[sample];
    return MLBM_OK;
}

mlbm_status mlbm_batch_permeability(mlbm_ctx* c, double* k, double* us, double* ui, double* tort) {
    if (!c) return set_error(MLBM_E_INVALID, "batch_permeability: NULL context");
    const int ns = (int)c->seg_off.size() - 1;
    std::vector<double> h(6 * (size_t)ns);
    MLBM_TRY(observe(c, kObserveFields, nullptr, nullptr));
    MLBM_TRY(read_results(c, h.data(), h.size()));
    for (int i = 0; i < ns; ++i) {
        const double* v = &h[6 * (size_t)i];
        const mlbm_params& p = c->seg_params[i];
        const double sup = v[2] / c->seg_box_area[i];
        const double gmag = std::sqrt(p.gx * p.gx + p.gy * p.gy);
        const double nu = (p.tau - 0.5) / 3.0;
        if (us) us[i] = sup;
        if (ui) ui[i] = v[0] != 0 ? v[2] / v[0] : 0.0;
        if (k) k[i] = gmag > 0 ? nu * sup / gmag : 0.0;
        if (tort) tort[i] = v[2] != 0 ? v[4] / v[2] : 0.0;
    }
    return MLBM_OK;
}

mlbm_status mlbm_batch_run_to_steady(mlbm_ctx* c, double tol, int64_t window, int64_t max_steps, int64_t* taken) {
    return mlbm_batch_run_to_steady_ex(c, tol, window, window, max_steps, taken);
}

mlbm_status mlbm_batch_run_to_steady_ex(mlbm_ctx* c, double tol, int64_t window, int64_t check, int64_t max_steps,
                                        int64_t* taken) {
    if (!c) return set_error(MLBM_E_INVALID, "batch_run_to_steady: NULL context");
    return run_steady(c, kFieldNorm, tol, window, check, max_steps, nullptr, taken, "batch_run_to_steady");
}

mlbm_status mlbm_batch_run_to_steady_mean(mlbm_ctx* c, double threshold, int64_t dn, int64_t check,
                                          const double* dt, int64_t max_steps, int64_t* taken) {
    if (!c) return set_error(MLBM_E_INVALID, "batch_run_to_steady_mean: NULL context");
    return run_steady(c, kMeanVelocity, threshold, dn, check, max_steps, dt, taken, "batch_run_to_steady_mean");
}

mlbm_status mlbm_batch_drag_lift(mlbm_ctx* c, const double* ref_length, const double* u_ref, double* fx, double* fy,
                                 double* cd, double* cl) {
    if (!c) return set_error(MLBM_E_INVALID, "batch_drag_lift: NULL context");
    const int ns = (int)c->seg_off.size() - 1;
    // link nodes are listed in position order and samples own contiguous
    // position ranges, so each sample's links are a contiguous slice
    const std::vector<int>& lo = c->link_off;
    for (int i = 0; i < ns; ++i) {
        const int m = lo[i + 1] - lo[i];
        if (m == 0) continue;
        MLBM_CUDA(launch_force(c->S, c->params.model, m, c->link_nodes + lo[i], c->area_over_s2, c->f8[c->cur],
                               c->ruv[c->cur], c->C, c->scratch, c->seg_out + 2 * i, c->stream));
    }
    std::vector<double> dv(2 * (size_t)ns);
    MLBM_TRY(read_results(c, dv.data(), dv.size()));
    for (int i = 0; i < ns; ++i) {
        const bool any = lo[i + 1] > lo[i];
        const double Fx = any ? dv[2 * i] : 0.0, Fy = any ? dv[2 * i + 1] : 0.0;
        if (fx) fx[i] = Fx;
        if (fy) fy[i] = Fy;
        const double sq = c->seg_s.empty() ? c->s : c->seg_s[i];
        const double L = ref_length ? ref_length[i] / sq : 0.0;
        const double u = u_ref ? u_ref[i] : 0.0;
        const double den = u * u * L;
        if (cd) cd[i] = den != 0 ? 2.0 * Fx / den : 0.0;
        if (cl) cl[i] = den != 0 ? 2.0 * Fy / den : 0.0;
    }
    return MLBM_OK;
}

mlbm_status mlbm_warm_start(mlbm_ctx* c, mlbm_mlp* m, const float* X, const double* scale_u,
                            const double* scale_rho, int* n_cold) {
    if (!c || !m || !X || !scale_u) return set_error(MLBM_E_INVALID, "warm_start: NULL argument");
    const int no = mlbm_mlp_outputs(m);
    if (no != 2 && no != 3) return set_error(MLBM_E_INVALID, "warm_start: the network must have 2 or 3 outputs");
    if (no == 3 && !scale_rho) return set_error(MLBM_E_INVALID, "warm_start: NULL density scale");
    const int ns = (int)c->seg_off.size() - 1;
    for (int i = 0; i < ns; ++i)
        if (!std::isfinite(scale_u[i]) || (no == 3 && !std::isfinite(scale_rho[i])))
            return set_error(MLBM_E_INVALID, "warm_start: non-finite scale");
    if (n_cold) *n_cold = 0;
    const int n = (int)c->n;
    // one temporary buffer: scales (2 ns doubles), density means (ns
    // doubles), flags (ns ints), then the prediction Y[n][no] (16-byte aligned)
    const size_t head = ((size_t)ns * 28 + 15) / 16 * 16;
    void* buf = nullptr;
    MLBM_CUDA(cudaMallocAsync(&buf, head + (size_t)n * no * sizeof(float) + 16, c->stream));
    double* dscale_u = static_cast<double*>(buf);
    double* dscale_r = dscale_u + ns;
    double* dmean = dscale_r + ns;
    int* flag = reinterpret_cast<int*>(dmean + ns);
    float* Y = reinterpret_cast<float*>(static_cast<char*>(buf) + head);
    // releases the temporary buffer (stream-ordered) and passes a status on
    auto release = [&](mlbm_status s) {
        cudaFreeAsync(buf, c->stream);
        return s;
    };
    std::vector<double> hs(2 * (size_t)ns, 0.0);
    for (int i = 0; i < ns; ++i) {
        hs[i] = scale_u[i];
        hs[ns + i] = no == 3 ? scale_rho[i] : 0.0;
    }
    cudaError_t e = cudaMemcpyAsync(dscale_u, hs.data(), 16 * (size_t)ns, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(flag, 0, (size_t)ns * 4, c->stream);
    if (e != cudaSuccess) return release(set_error(MLBM_E_CUDA, std::string("warm_start: ") + cudaGetErrorString(e)));
    mlbm_status st = mlbm_mlp_forward_device(m, X, n, Y, c->stream);
    if (st != MLBM_OK) return release(st);
    e = launch_warm_check(n, c->perm, c->S.node_sample, c->meta, Y, no, dscale_u, dscale_r, 0.3f, 0.1f, flag,
                          c->stream);
    if (e == cudaSuccess && no == 3) {
        // area-weighted mean of the predicted density deviation per sample
        e = launch_warm_drho(n, c->perm, c->S.node_sample, c->meta, Y, no, dscale_r, c->rho, c->stream);
        if (e == cudaSuccess)
            e = launch_warm_means(ns, c->max_blocks, c->seg_dev, c->rho, c->area, c->mask, c->scratch, dmean,
                                  c->stream);
    }
    if (e == cudaSuccess)
        e = launch_warm_fill(n, c->perm, c->S.node_sample, c->meta, c->eqv, Y, no, dscale_u, c->rho, dmean, flag, c->io,
                             c->stream);
    if (e == cudaSuccess) {
        if (c->params.model == MLBM_MODEL_BGK)
            e = launch_set_bgk_equilibrium(n, c->perm, c->io, c->f8[c->cur], c->f0[c->cur], c->stream);
        else
            e = launch_set_tau1(n, c->perm, c->io, c->ruv[c->cur], c->stream);
    }
    std::vector<int> hflag(ns, 0);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hflag.data(), flag, (size_t)ns * 4, cudaMemcpyDeviceToHost, c->stream);
    if (e != cudaSuccess) return release(set_error(MLBM_E_CUDA, std::string("warm_start: ") + cudaGetErrorString(e)));
    MLBM_TRY(release(MLBM_OK));
    MLBM_TRY(sync(c));
    if (n_cold)
        for (int i = 0; i < ns; ++i) *n_cold += hflag[i] != 0;
    c->steps = 0;
    return MLBM_OK;
}

mlbm_status mlbm_autotune_order(mlbm_stencils* const* sts, const mlbm_params* params, int n_samples,
                                int steps_per_variant, int flush_l2, int* best_order, int* best_variant,
                                double* best_ms) {
    clear_error();
    if (!sts || !params || n_samples < 1 || steps_per_variant < 1)
        return set_error(MLBM_E_INVALID, "autotune_order: bad arguments");
    int bo = -1, bv = -1;
    double bt = 1e300;
    for (int order = MLBM_ORDER_HILBERT; order <= MLBM_ORDER_INPUT; ++order) {
        for (int i = 0; i < n_samples; ++i) MLBM_TRY(mlbm_stencils_set_order(sts[i], order));
        mlbm_ctx* c = nullptr;
        mlbm_status st = n_samples == 1 ? mlbm_init(&c, sts[0], &params[0], nullptr, nullptr)
                                        : mlbm_batch_init(&c, sts, params, n_samples);
        if (st != MLBM_OK) return st;
        double ms = 0.0;
        st = mlbm_autotune_ex(c, steps_per_variant, flush_l2, &ms);
        const int v = c->variant;
        mlbm_destroy(c);
        if (st != MLBM_OK) return st;
        if (ms < bt) {
            bt = ms;
            bo = order;
            bv = v;
        }
    }
    for (int i = 0; i < n_samples; ++i) MLBM_TRY(mlbm_stencils_set_order(sts[i], bo));
    if (best_order) *best_order = bo;
    if (best_variant) *best_variant = bv;
    if (best_ms) *best_ms = bt;
    return MLBM_OK;
}

mlbm_status mlbm_set_graphs(mlbm_ctx* c, int enable) {
    if (!c) return set_error(MLBM_E_INVALID, "set_graphs: NULL context");
    c->use_graphs = enable != 0;
    if (!c->use_graphs) drop_graphs(c);
    return MLBM_OK;
}

int64_t mlbm_reduce_scratch_doubles(int64_t n) { return n < 0 ? -1 : 6 * (int64_t)reduce_blocks(n); }

mlbm_status mlbm_reduce_fields_device(const float* rho, const float* ux, const float* uy, const float* area,
                                      const uint8_t* mask, int64_t n, double* scratch, int64_t scratch_len,
                                      double* out, void* stream) {
    clear_error();
    // the node arrays may be NULL when there are no nodes
    if ((n > 0 && (!rho || !ux || !uy || !area)) || !scratch || !out || n < 0)
        return set_error(MLBM_E_INVALID, "reduce_fields_device: NULL pointer or negative n");
    if (scratch_len < mlbm_reduce_scratch_doubles(n))
        return set_error(MLBM_E_INVALID, "reduce_fields_device: scratch too small");
    MLBM_CUDA(launch_reduce_fields(rho, ux, uy, area, mask, n, scratch, out, static_cast<cudaStream_t>(stream)));
    return MLBM_OK;
}

// ------------------------------------------------------ partitioned step
// P logical partitions of one node set, each a context over a contiguous
// range of the device positions with halo slots after its own nodes.  In a
// step every partition reads its own buffers only, and the new states of the
// nodes that another partition references go into that partition's halo slots
// of the buffer being written.  With kernel variants 27..29 all partitions
// step in one launch whose threads store those states themselves; with any
// other variant each partition is launched in turn and one kernel then copies
// the states.  Steps are replayed from captured graphs of kGraphSteps.  (Four
// partitions of 96k nodes, tau = 1: 110 us a step with a launch per partition
// and a packing kernel and a copy per pair of partitions, 9.5 us now.)
}  // extern "C"

struct mlbm_part {
    int P = 0;
    int model = 0;
    int64_t n = 0;
    double box_area = 1.0;
    std::vector<mlbm_ctx*> ctx;
    std::vector<int64_t> first, n_owned, n_halo;
    // device: the partitions, the step's blocks as (partition, range), the
    // halo entries (owner, position, receiver, slot), the FP64 I/O array of
    // all nodes in the caller's order, and the partitions' error words
    dev::PartDev* parts = nullptr;
    int2* work = nullptr;
    int blocks = 0;
    int4* halo = nullptr;
    int64_t n_copies = 0;
    double* io = nullptr;
    int* err = nullptr;
    cudaStream_t stream = nullptr;
    cudaGraphExec_t graph[2] = {nullptr, nullptr};  // kGraphSteps steps from buffer 0 / 1
    int graph_variant = -1;
    std::vector<void*> allocations;
    int64_t steps = 0;
};

namespace {

void drop_part_graphs(mlbm_part* P) {
    for (cudaGraphExec_t& g : P->graph) {
        if (g) cudaGraphExecDestroy(g);
        g = nullptr;
    }
    P->graph_variant = -1;
}

void free_part(mlbm_part* P) {
    if (!P) return;
    if (P->stream) cudaStreamSynchronize(P->stream);
    drop_part_graphs(P);
    for (mlbm_ctx* c : P->ctx) free_ctx(c);
    for (void* q : P->allocations) cudaFree(q);
    if (P->stream) cudaStreamDestroy(P->stream);
    delete P;
}

int state_width(const mlbm_part* P) { return P->model == MLBM_MODEL_BGK ? 2 : 1; }

template <class T>
mlbm_status part_alloc(mlbm_part* P, T** dst, size_t count) {
    void* d = nullptr;
    if (cudaMalloc(&d, std::max<size_t>(count, 1) * sizeof(T)) != cudaSuccess) {
        (void)cudaGetLastError();
        return set_error(MLBM_E_OOM, "part_init: cudaMalloc");
    }
    P->allocations.push_back(d);
    *dst = static_cast<T*>(d);
    return MLBM_OK;
}

template <class T>
mlbm_status part_upload(mlbm_part* P, T** dst, const std::vector<T>& src) {
    MLBM_TRY(part_alloc(P, dst, src.size()));
    MLBM_CUDA(cudaMemcpyAsync(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, P->stream));
    MLBM_CUDA(cudaStreamSynchronize(P->stream));
    return MLBM_OK;
}

// fill every partition's halo slots from the owners' current states
mlbm_status exchange(mlbm_part* P) {
    MLBM_CUDA(launch_exchange(P->parts, P->halo, P->n_copies, state_width(P), P->ctx[0]->cur, P->stream));
    return MLBM_OK;
}

mlbm_status part_sync(mlbm_part* P) {
    std::vector<int> e(P->P, 0);
    MLBM_CUDA(cudaMemcpyAsync(e.data(), P->err, e.size() * sizeof(int), cudaMemcpyDeviceToHost, P->stream));
    MLBM_CUDA(cudaStreamSynchronize(P->stream));
    for (mlbm_ctx* c : P->ctx)
        if (e[(size_t)(c->err - P->err)] != 0) return sync(c);  // clears the word and reports it
    return MLBM_OK;
}

// one step of every partition on the stream
mlbm_status part_launch_step(mlbm_part* P) {
    mlbm_ctx* c0 = P->ctx[0];
    if (c0->variant >= 27 && c0->variant <= 29 && c0->S.rec) {
        const dev::Wait W{c0->wait_ns, 0};
        MLBM_CUDA(launch_step_parts(P->model == MLBM_MODEL_BGK ? 0 : 1, c0->S.Kq, P->n, P->parts, P->work, P->blocks,
                                    c0->cur, P->err, W, P->stream));
        for (mlbm_ctx* c : P->ctx) c->cur ^= 1;
        return MLBM_OK;
    }
    for (mlbm_ctx* c : P->ctx) MLBM_TRY(launch_one_step(c, c->variant));
    return exchange(P);
}

// instantiate the graph of kGraphSteps steps from buffer `parity`
mlbm_status part_graph(mlbm_part* P, int parity) {
    if (P->graph[parity]) return MLBM_OK;
    cudaGraph_t g = nullptr;
    const int cur = P->ctx[0]->cur;
    MLBM_CUDA(cudaStreamBeginCapture(P->stream, cudaStreamCaptureModeThreadLocal));
    for (mlbm_ctx* c : P->ctx) c->cur = parity;
    mlbm_status s = MLBM_OK;
    for (int i = 0; i < kGraphSteps && s == MLBM_OK; ++i) s = part_launch_step(P);
    cudaError_t e = cudaStreamEndCapture(P->stream, &g);
    for (mlbm_ctx* c : P->ctx) c->cur = cur;
    if (s == MLBM_OK && e == cudaSuccess) e = cudaGraphInstantiate(&P->graph[parity], g, 0);
    if (g) cudaGraphDestroy(g);
    if (s != MLBM_OK) return s;
    if (e != cudaSuccess) {
        P->graph[parity] = nullptr;
        return set_error(MLBM_E_CUDA, std::string("part_step: graph: ") + cudaGetErrorString(e));
    }
    return MLBM_OK;
}

}  // namespace

extern "C" {

mlbm_status mlbm_part_init(mlbm_part** out, const mlbm_stencils* st, const mlbm_params* p, int n_parts,
                           const int64_t* bounds) {
    clear_error();
    if (!out || !st || !p) return set_error(MLBM_E_INVALID, "part_init: NULL argument");
    *out = nullptr;
    MLBM_TRY(check_params(p));
    if (st->h.n > (int64_t(1) << 31) - 1) return set_error(MLBM_E_INVALID, "part_init: too many nodes");
    PartPlan plan;
    MLBM_TRY(make_part_plan(st->h, n_parts, bounds, plan));
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
        (void)cudaGetLastError();
        return set_error(MLBM_E_CUDA, "part_init: no CUDA device");
    }
    auto* P = new (std::nothrow) mlbm_part;
    if (!P) return set_error(MLBM_E_OOM, "part_init: out of host memory");
    P->P = n_parts;
    P->model = p->model;
    P->n = st->h.n;
    P->box_area = st->h.box_area;
    auto fail = [&](mlbm_status s) {
        std::string msg = g_last_error;
        free_part(P);
        return set_error(s, msg);
    };
    if (cudaStreamCreateWithFlags(&P->stream, cudaStreamNonBlocking) != cudaSuccess)
        return fail(set_error(MLBM_E_CUDA, "part_init: stream"));
    for (int q = 0; q < n_parts; ++q) {
        auto* sub = new (std::nothrow) mlbm_stencils;
        if (!sub) return fail(set_error(MLBM_E_OOM, "part_init: out of host memory"));
        sub->h = slice_partition(st->h, plan, q);
        auto* c = new (std::nothrow) mlbm_ctx;
        if (!c) {
            delete sub;
            return fail(set_error(MLBM_E_OOM, "part_init: out of host memory"));
        }
        P->ctx.push_back(c);
        mlbm_status s = do_init(c, sub, p, nullptr, nullptr);
        delete sub;
        if (s != MLBM_OK) return fail(s);
        c->stream = P->stream;
        c->use_graphs = false;
        const int64_t a = plan.bounds[q], e = plan.bounds[q + 1];
        P->first.push_back(a);
        P->n_owned.push_back(e - a);
        P->n_halo.push_back((int64_t)plan.halo[q].size());
        // I/O goes through one array of all nodes in the caller's order
        std::vector<int> ids((size_t)c->n_pad, 0);
        for (int64_t i = a; i < e; ++i) ids[(size_t)(i - a)] = (int)st->h.perm[i];
        if (cudaMemcpyAsync(c->perm, ids.data(), ids.size() * sizeof(int), cudaMemcpyHostToDevice, P->stream) !=
                cudaSuccess ||
            cudaStreamSynchronize(P->stream) != cudaSuccess)
            return fail(set_error(MLBM_E_CUDA, "part_init: upload"));
    }
    // halo copies, and per owner the slots each of its nodes is sent to
    std::vector<int4> halo;
    std::vector<std::vector<std::pair<int, int2>>> sends(n_parts);
    for (int q = 0; q < n_parts; ++q)
        for (int o = 0; o < n_parts; ++o)
            for (int64_t i = plan.halo_off[q][o]; i < plan.halo_off[q][o + 1]; ++i) {
                const int pos = (int)(plan.halo[q][(size_t)i] - plan.bounds[o]), slot = (int)(P->n_owned[q] + i);
                halo.push_back(make_int4(o, pos, q, slot));
                sends[o].push_back({pos, make_int2(q, slot)});
            }
    P->n_copies = (int64_t)halo.size();
    mlbm_status us = part_upload(P, &P->halo, halo);
    if (us == MLBM_OK) us = part_alloc(P, &P->io, 9 * (size_t)P->n);
    if (us == MLBM_OK) us = part_upload(P, &P->err, std::vector<int>(n_parts, 0));
    if (us != MLBM_OK) return fail(us);
    // the step's blocks, shared out by node count
    const int sms = warp_step_ranges(1 << 30);
    std::vector<dev::PartDev> dev_parts(n_parts);
    std::vector<int2> work;
    for (int q = 0; q < n_parts; ++q) {
        mlbm_ctx* c = P->ctx[q];
        c->err = P->err + q;
        std::stable_sort(sends[q].begin(), sends[q].end(),
                         [](const auto& x, const auto& y) { return x.first < y.first; });
        std::vector<int> send_first((size_t)c->n + 1, 0);
        std::vector<int2> to;
        for (const auto& e : sends[q]) {
            ++send_first[(size_t)e.first + 1];
            to.push_back(e.second);
        }
        for (int64_t i = 0; i < c->n; ++i) send_first[(size_t)i + 1] += send_first[(size_t)i];
        dev::PartDev& D = dev_parts[q];
        int* d_first = nullptr;
        int2* d_to = nullptr;
        us = part_upload(P, &d_first, send_first);
        if (us == MLBM_OK) us = part_upload(P, &d_to, to);
        if (us != MLBM_OK) return fail(us);
        const int64_t lo = sms * P->first[q] / P->n, hi = sms * (P->first[q] + P->n_owned[q]) / P->n;
        c->S.n_ranges = (int)std::max<int64_t>(1, std::min<int64_t>({hi - lo, (c->n + 31) / 32, c->S.n_ranges}));
        for (int r = 0; r < c->S.n_ranges; ++r) work.push_back(make_int2(q, r));
        cudaError_t e = launch_mark_sends((int)c->n, d_first, c->meta, P->stream);
        if (e == cudaSuccess) e = launch_record_kinds(c->S, c->rec, c->need, c->range, P->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(P->stream);
        if (e != cudaSuccess) return fail(set_error(MLBM_E_CUDA, "part_init: kinds"));
        D.S = c->S;
        D.C = c->C;
        for (int b = 0; b < 2; ++b) {
            D.state[b] = c->f8[b] ? c->f8[b] : c->ruv[b];
            D.f0[b] = c->f0[b];
        }
        D.send_first = d_first;
        D.sends = d_to;
    }
    P->blocks = (int)work.size();
    us = part_upload(P, &P->parts, dev_parts);
    if (us == MLBM_OK) us = part_upload(P, &P->work, work);
    if (us != MLBM_OK) return fail(us);
    mlbm_status s = exchange(P);
    if (s == MLBM_OK) s = part_sync(P);
    P->graph_variant = P->ctx[0]->variant;
    if (s == MLBM_OK) s = part_graph(P, 0);  // the one from buffer 1 when steps first start there
    if (s != MLBM_OK) return fail(s);
    *out = P;
    return MLBM_OK;
}

void mlbm_part_destroy(mlbm_part* P) { free_part(P); }

mlbm_status mlbm_part_info(const mlbm_part* P, int part, int64_t* first, int64_t* n_owned, int64_t* n_halo,
                           int64_t* halo_bytes_per_step) {
    if (!P || part < 0 || part >= P->P) return set_error(MLBM_E_INVALID, "part_info: bad argument");
    if (first) *first = P->first[part];
    if (n_owned) *n_owned = P->n_owned[part];
    if (n_halo) *n_halo = P->n_halo[part];
    if (halo_bytes_per_step) *halo_bytes_per_step = P->n_halo[part] * state_width(P) * (int64_t)sizeof(float4);
    return MLBM_OK;
}

mlbm_status mlbm_part_set_kernel_variant(mlbm_part* P, int variant) {
    if (!P) return set_error(MLBM_E_INVALID, "part_set_kernel_variant: NULL");
    for (mlbm_ctx* c : P->ctx) MLBM_TRY(mlbm_set_kernel_variant(c, variant));
    return MLBM_OK;
}

mlbm_status mlbm_part_step(mlbm_part* P, int64_t n_steps) {
    if (!P) return set_error(MLBM_E_INVALID, "part_step: NULL");
    if (n_steps < 0) return set_error(MLBM_E_INVALID, "part_step: negative step count");
    int64_t left = n_steps;
    if (n_steps >= kGraphSteps) {
        if (P->graph_variant != P->ctx[0]->variant) {
            drop_part_graphs(P);
            P->graph_variant = P->ctx[0]->variant;
        }
        for (; left >= kGraphSteps; left -= kGraphSteps) {
            MLBM_TRY(part_graph(P, P->ctx[0]->cur));
            MLBM_CUDA(cudaGraphLaunch(P->graph[P->ctx[0]->cur], P->stream));
        }
    }
    for (; left > 0; --left) MLBM_TRY(part_launch_step(P));
    for (mlbm_ctx* c : P->ctx) c->steps += n_steps;
    P->steps += n_steps;
    return part_sync(P);  // also reports a bounded wait that ran out
}

// fields or populations in the caller's order for all nodes; `width` values per node
static mlbm_status part_set(mlbm_part* P, const double* v, int width, bool fields) {
    MLBM_CUDA(cudaMemcpyAsync(P->io, v, (size_t)P->n * width * 8, cudaMemcpyHostToDevice, P->stream));
    for (mlbm_ctx* c : P->ctx) {
        const int n = (int)c->n, b = c->cur;
        if (!fields) MLBM_CUDA(launch_set_bgk(n, c->perm, P->io, c->f8[b], c->f0[b], P->stream));
        else if (P->model == MLBM_MODEL_BGK)
            MLBM_CUDA(launch_set_bgk_equilibrium(n, c->perm, P->io, c->f8[b], c->f0[b], P->stream));
        else MLBM_CUDA(launch_set_tau1(n, c->perm, P->io, c->ruv[b], P->stream));
        c->steps = 0;
    }
    MLBM_TRY(exchange(P));
    P->steps = 0;
    return part_sync(P);
}

static mlbm_status part_get(mlbm_part* P, double* v, int width, bool fields) {
    for (mlbm_ctx* c : P->ctx) {
        if (fields) MLBM_TRY(fields_to(c, P->io, 0));
        else MLBM_CUDA(launch_get_bgk((int)c->n, c->perm, c->f8[c->cur], c->f0[c->cur], P->io, P->stream));
    }
    MLBM_CUDA(cudaMemcpyAsync(v, P->io, (size_t)P->n * width * 8, cudaMemcpyDeviceToHost, P->stream));
    return part_sync(P);
}

mlbm_status mlbm_part_set_fields(mlbm_part* P, const double* ru) {
    if (!P || !ru) return set_error(MLBM_E_INVALID, "part_set_fields: NULL argument");
    return part_set(P, ru, 3, true);
}

mlbm_status mlbm_part_get_fields(mlbm_part* P, double* ru) {
    if (!P || !ru) return set_error(MLBM_E_INVALID, "part_get_fields: NULL argument");
    return part_get(P, ru, 3, true);
}

mlbm_status mlbm_part_set_populations(mlbm_part* P, const double* f) {
    if (!P || !f) return set_error(MLBM_E_INVALID, "part_set_populations: NULL argument");
    if (P->model != MLBM_MODEL_BGK) return set_error(MLBM_E_INVALID, "part_set_populations: BGK only");
    return part_set(P, f, 9, false);
}

mlbm_status mlbm_part_get_populations(mlbm_part* P, double* f) {
    if (!P || !f) return set_error(MLBM_E_INVALID, "part_get_populations: NULL argument");
    if (P->model != MLBM_MODEL_BGK) return set_error(MLBM_E_INVALID, "part_get_populations: BGK only");
    return part_get(P, f, 9, false);
}

mlbm_status mlbm_part_permeability(mlbm_part* P, double* k, double* us, double* ui, double* tort) {
    if (!P) return set_error(MLBM_E_INVALID, "part_permeability: NULL");
    // each partition's six FP64 sums, then added in partition order (the
    // all-reduce of a run whose partitions live on separate devices)
    double tot[6] = {0, 0, 0, 0, 0, 0};
    for (mlbm_ctx* c : P->ctx) {
        double h[6];
        MLBM_TRY(sums_of_all(c, h));
        for (int i = 0; i < 6; ++i) tot[i] += h[i];
    }
    const mlbm_params& pp = P->ctx[0]->params;
    const double sup = tot[2] / P->box_area;
    const double gmag = std::sqrt(pp.gx * pp.gx + pp.gy * pp.gy);
    const double nu = (pp.tau - 0.5) / 3.0;
    if (us) *us = sup;
    if (ui) *ui = tot[0] != 0 ? tot[2] / tot[0] : 0.0;
    if (k) *k = gmag > 0 ? nu * sup / gmag : 0.0;
    if (tort) *tort = tot[2] != 0 ? tot[4] / tot[2] : 0.0;
    return MLBM_OK;
}

}  // extern "C"
