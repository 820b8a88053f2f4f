// Lattice LBM on a regular nx x ny grid: the comparison method of the paper
// (Sec. 2.1, Eq. (1)-(3): streaming by one lattice spacing per step, then
// collision), with the same FP32 collision as the meshless step (shifted
// populations g = f - w, TRT/BGK with the second-order source, conservative
// pair form).  Cells are fluid, solid (half-way bounce-back on the links
// that come from a solid cell: g_k(x) = g*_k'(x)) or equilibrium (g =
// g^eq(rho_b, u_b) every step).  Layout: one plane of n = nx ny floats per
// population (k = 0..8), row-major cells, two buffers; a step is one pull
// kernel, thread per cell, replayed from captured graphs.
#include <cmath>
#include <string>
#include <vector>

#include "kernels.h"
#include "launch_util.cuh"
#include "mlbm_internal.h"
#include "step_node.cuh"

namespace mlbm {
namespace dev {

enum : uint8_t { kCellFluid = 0, kCellSolid = 1, kCellEq = 2 };
// what a cell does in a step, worked out once: bits 0..7 direction k = 1..8
// bounces back (its source is solid or outside a non-periodic side), and
constexpr uint16_t kInfoSolid = 0x100, kInfoEq = 0x200;

// One thread per cell.  The step is bound by the 73 bytes a cell moves through
// L2 or HBM, so everything else is kept off the load path: one info word per
// cell (read before the previous step has finished) instead of the types of
// nine cells and the wrap-around divisions, all nine populations loaded at
// once, and the rare bounced ones fetched again from the cell itself.  Rows of
// 64 cells by 4 fill narrow lattices too.  577,280 cells (42 MB, in L2), us a
// step: 14.3 with the types of nine cells and a launch per step, 9.3 now.
constexpr int kLatX = 64, kLatY = 4;
__global__ void __launch_bounds__(kLatX * kLatY) lattice_step(int nx, int ny, const uint16_t* __restrict__ info,
                                                              const float4* __restrict__ eqv,
                                                              const float* __restrict__ fin, float* __restrict__ fout,
                                                              Collide C) {
    const int x = blockIdx.x * kLatX + threadIdx.x, y = blockIdx.y * kLatY + threadIdx.y;
    const size_t n = (size_t)nx * ny;
    const size_t i = (size_t)y * nx + x;
    const uint16_t c = x < nx && y < ny ? info[i] : kInfoSolid;
    pdl_trigger();
    pdl_wait();
    if (c & kInfoSolid) return;
    float g[9];
    if (c & kInfoEq) {
        const float4 e = eqv[i];
        eq_populations(e.x, e.y, e.z, g);
    } else {
        const int dxm = x > 0 ? -1 : nx - 1, dxp = x + 1 < nx ? 1 : 1 - nx;
        const long long dym = y > 0 ? -(long long)nx : (long long)(ny - 1) * nx;
        const long long dyp = y + 1 < ny ? (long long)nx : -(long long)(ny - 1) * nx;
        g[0] = fin[i];
#pragma unroll
        for (int k = 1; k < 9; ++k) {
            const long long d = (ex_of(k) > 0 ? dxm : (ex_of(k) < 0 ? dxp : 0)) +
                                (ey_of(k) > 0 ? dym : (ey_of(k) < 0 ? dyp : 0LL));
            g[k] = fin[(size_t)k * n + (size_t)((long long)i + d)];
        }
        if (c & 0xff) {
#pragma unroll
            for (int k = 1; k < 9; ++k)
                if ((c >> (k - 1)) & 1) g[k] = fin[(size_t)opp_of(k) * n + i];
        }
        collide_pairs(g, C, 0xFu, true);
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) fout[(size_t)k * n + i] = g[k];
}

// momentum exchange on the bounce-back links of the state `st` (post
// collision): a link (x, k) whose source x - e_k is solid receives
// g*_k'(x), and the body takes 2 g*_k'(x) e_k' (populations relative to the
// rest state, as for the meshless wall force).  One block over the fluid
// cells with such links (listed once), FP64 sums in a fixed order: a call took
// 64 us when it looked over all 577,280 cells for them.
__global__ void __launch_bounds__(256) lattice_force(size_t n, int m, const int2* __restrict__ wall,
                                                     const float* __restrict__ st, double* __restrict__ out) {
    double fx = 0.0, fy = 0.0;
    for (int e = threadIdx.x; e < m; e += 256) {
        const int2 w = wall[e];  // cell, solid links as in the info word
#pragma unroll
        for (int k = 1; k < 9; ++k) {
            if (!((w.y >> (k - 1)) & 1)) continue;
            const int kp = opp_of(k);
            const double v = st[(size_t)kp * n + w.x];
            fx += 2.0 * v * ex_of(kp);
            fy += 2.0 * v * ey_of(kp);
        }
    }
    __shared__ double sx_[256], sy_[256];
    sx_[threadIdx.x] = fx;
    sy_[threadIdx.x] = fy;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) {
            sx_[threadIdx.x] += sx_[threadIdx.x + h];
            sy_[threadIdx.x] += sy_[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = sx_[0];
        out[1] = sy_[0];
    }
}

// populations (FP64, [n][9], unshifted) <-> state planes (FP32, shifted)
__global__ void lattice_set(size_t n, const double* __restrict__ f, float* __restrict__ st) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
#pragma unroll
    for (int k = 0; k < 9; ++k) st[(size_t)k * n + i] = (float)(f[9 * i + k] - (double)w_of(k));
}

__global__ void lattice_get(size_t n, const float* __restrict__ st, double* __restrict__ f) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
#pragma unroll
    for (int k = 0; k < 9; ++k) f[9 * i + k] = (double)st[(size_t)k * n + i] + (double)w_of(k);
}

}  // namespace dev
}  // namespace mlbm

using namespace mlbm;

struct mlbm_lattice {
    int nx = 0, ny = 0, px = 0, py = 0;
    mlbm_params params{};
    dev::Collide C{};
    uint16_t* info = nullptr;
    int2* wall = nullptr;  // cells with solid links
    int n_wall = 0;
    float4* eqv = nullptr;
    float* f[2] = {nullptr, nullptr};
    double* io = nullptr;
    double* small = nullptr;
    int cur = 0;
    int64_t steps = 0;
    cudaStream_t stream = nullptr;
    cudaGraphExec_t graph[2] = {nullptr, nullptr};  // kLatGraph steps from buffer 0 / 1
};

namespace {
#define LAT_CUDA(call)                                                                                        \
    do {                                                                                                      \
        cudaError_t e_ = (call);                                                                              \
        if (e_ != cudaSuccess) return set_error(MLBM_E_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)
constexpr int kLatGraph = 16;  // steps of a captured graph (even: it ends on the buffer it starts from)

void free_lattice(mlbm_lattice* L) {
    if (!L) return;
    if (L->stream) cudaStreamSynchronize(L->stream);
    for (cudaGraphExec_t g : L->graph)
        if (g) cudaGraphExecDestroy(g);
    cudaFree(L->info);
    cudaFree(L->wall);
    cudaFree(L->eqv);
    cudaFree(L->f[0]);
    cudaFree(L->f[1]);
    cudaFree(L->io);
    cudaFree(L->small);
    if (L->stream) cudaStreamDestroy(L->stream);
    delete L;
}

// one step from the current buffer into the other, overlapping the launch
// with the step before
cudaError_t launch_lattice_step(mlbm_lattice* L) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((L->nx + dev::kLatX - 1) / dev::kLatX, (L->ny + dev::kLatY - 1) / dev::kLatY);
    cfg.blockDim = dim3(dev::kLatX, dev::kLatY);
    cfg.stream = L->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e =
        cudaLaunchKernelEx(&cfg, dev::lattice_step, L->nx, L->ny, (const uint16_t*)L->info, (const float4*)L->eqv,
                           (const float*)L->f[L->cur], L->f[1 - L->cur], L->C);
    L->cur = 1 - L->cur;
    return e;
}

// the graph of kLatGraph steps that starts from buffer `from`
cudaError_t capture_lattice(mlbm_lattice* L, int from) {
    cudaGraph_t g = nullptr;
    const int cur = L->cur;
    cudaError_t e = cudaStreamBeginCapture(L->stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    L->cur = from;
    for (int i = 0; i < kLatGraph && e == cudaSuccess; ++i) e = launch_lattice_step(L);
    const cudaError_t ee = cudaStreamEndCapture(L->stream, &g);
    L->cur = cur;
    if (e == cudaSuccess) e = ee;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&L->graph[from], g, 0);
    if (e != cudaSuccess) L->graph[from] = nullptr;
    if (g) cudaGraphDestroy(g);
    return e;
}
}  // namespace

extern "C" {

mlbm_status mlbm_lattice_init(mlbm_lattice** out, int nx, int ny, int periodic_x, int periodic_y,
                              const uint8_t* cell, const double* eq_values, const mlbm_params* p) {
    clear_error();
    // rows map to the grid's y dimension (at most 65535)
    if (!out || !cell || !p || nx < 1 || ny < 1 || ny > 65535 || (int64_t)nx * ny > (int64_t(1) << 31) - 1)
        return set_error(MLBM_E_INVALID, "lattice_init: bad arguments (1 <= ny <= 65535, nx ny < 2^31)");
    *out = nullptr;
    if (p->model != MLBM_MODEL_BGK || !(p->tau > 0.5) || (p->tau_minus > 0 && !(p->tau_minus > 0.5)) ||
        !std::isfinite(p->gx) || !std::isfinite(p->gy))
        return set_error(MLBM_E_INVALID, "lattice_init: BGK/TRT parameters with tau > 1/2 needed");
    const size_t n = (size_t)nx * ny;
    bool has_eq = false;
    for (size_t i = 0; i < n; ++i) {
        if (cell[i] > 2) return set_error(MLBM_E_INVALID, "lattice_init: cell types are 0, 1, 2");
        has_eq |= cell[i] == 2;
    }
    if (has_eq && !eq_values) return set_error(MLBM_E_INVALID, "lattice_init: equilibrium cells need eq_values");
    auto* L = new (std::nothrow) mlbm_lattice;
    if (!L) return set_error(MLBM_E_OOM, "lattice_init: out of host memory");
    L->nx = nx;
    L->ny = ny;
    L->px = periodic_x != 0;
    L->py = periodic_y != 0;
    L->params = *p;
    const double tp = p->tau, tm = p->tau_minus > 0 ? p->tau_minus : p->tau;
    L->C.omega_p = (float)(1.0 / tp);
    L->C.omega_m = (float)(1.0 / tm);
    L->C.src_p = (float)(1.0 - 0.5 / tp);
    L->C.src_m = (float)(1.0 - 0.5 / tm);
    L->C.ax = (float)p->gx;
    L->C.ay = (float)p->gy;
    std::vector<float4> he(n, make_float4(0, 0, 0, 0));
    if (eq_values)
        for (size_t i = 0; i < n; ++i)
            if (cell[i] == 2)
                he[i] = make_float4((float)(eq_values[3 * i] - 1.0), (float)eq_values[3 * i + 1],
                                    (float)eq_values[3 * i + 2], 0.f);
    // what each cell does in a step, and the cells with solid links in cell
    // order; the rows on all cores
    std::vector<uint16_t> info(n, 0);
    std::vector<std::vector<int2>> row_wall((size_t)ny);
#pragma omp parallel for schedule(static, 8)
    for (int y = 0; y < ny; ++y) {
        static const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
        // the rows that populations with e_y = -1, 0, 1 come from, and those outside
        const int sy[3] = {y + 1 < ny ? y + 1 : 0, y, y > 0 ? y - 1 : ny - 1};
        const bool out_y[3] = {!L->py && y + 1 == ny, false, !L->py && y == 0};
        for (int x = 0; x < nx; ++x) {
            const size_t i = (size_t)y * nx + x;
            if (cell[i] != dev::kCellFluid) {
                info[i] = cell[i] == dev::kCellSolid ? dev::kInfoSolid : dev::kInfoEq;
                continue;
            }
            const int sx[3] = {x + 1 < nx ? x + 1 : 0, x, x > 0 ? x - 1 : nx - 1};
            const bool out_x[3] = {!L->px && x + 1 == nx, false, !L->px && x == 0};
            int bounce = 0, solid = 0;
            for (int k = 1; k < 9; ++k) {
                const int a = ex[k] + 1, b = ey[k] + 1;
                if (out_x[a] || out_y[b]) bounce |= 1 << (k - 1);
                else if (cell[(size_t)sy[b] * nx + sx[a]] == dev::kCellSolid) solid |= 1 << (k - 1);
            }
            info[i] = (uint16_t)(bounce | solid);
            if (solid) row_wall[(size_t)y].push_back(make_int2((int)i, solid));
        }
    }
    std::vector<int2> wall;
    for (const auto& r : row_wall) wall.insert(wall.end(), r.begin(), r.end());
    L->n_wall = (int)wall.size();
    cudaError_t e = cudaStreamCreateWithFlags(&L->stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaMalloc(&L->info, n * sizeof(uint16_t));
    if (e == cudaSuccess && !wall.empty()) e = cudaMalloc(&L->wall, wall.size() * sizeof(int2));
    if (e == cudaSuccess) e = cudaMalloc(&L->eqv, n * sizeof(float4));
    if (e == cudaSuccess) e = cudaMalloc(&L->f[0], 9 * n * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&L->f[1], 9 * n * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&L->io, 9 * n * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&L->small, 2 * sizeof(double));
    if (e == cudaSuccess) e = cudaMemcpy(L->info, info.data(), n * sizeof(uint16_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !wall.empty())
        e = cudaMemcpy(L->wall, wall.data(), wall.size() * sizeof(int2), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(L->eqv, he.data(), n * sizeof(float4), cudaMemcpyHostToDevice);
    // rest state (shifted populations zero), equilibrium cells at their values
    if (e == cudaSuccess) e = cudaMemset(L->f[0], 0, 9 * n * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(L->f[1], 0, 9 * n * sizeof(float));
    // steps run on a stream that does not wait for the default stream's work
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
    if (e == cudaSuccess) e = capture_lattice(L, 0);  // the one from buffer 1 when steps first start there
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        free_lattice(L);
        return set_error(MLBM_E_CUDA, std::string("lattice_init: ") + cudaGetErrorString(e));
    }
    *out = L;
    return MLBM_OK;
}

void mlbm_lattice_destroy(mlbm_lattice* L) { free_lattice(L); }

mlbm_status mlbm_lattice_step(mlbm_lattice* L, int64_t n_steps) {
    if (!L || n_steps < 0) return set_error(MLBM_E_INVALID, "lattice_step: bad arguments");
    int64_t left = n_steps;
    for (; left >= kLatGraph; left -= kLatGraph) {
        if (!L->graph[L->cur]) LAT_CUDA(capture_lattice(L, L->cur));
        LAT_CUDA(cudaGraphLaunch(L->graph[L->cur], L->stream));
    }
    for (; left > 0; --left) LAT_CUDA(launch_lattice_step(L));
    L->steps += n_steps;
    return MLBM_OK;
}

mlbm_status mlbm_lattice_time_steps(mlbm_lattice* L, int64_t n_steps, double* ms) {
    if (!L || n_steps < 1 || !ms) return set_error(MLBM_E_INVALID, "lattice_time_steps: bad arguments");
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    LAT_CUDA(cudaEventCreate(&e0));
    LAT_CUDA(cudaEventCreate(&e1));
    cudaEventRecord(e0, L->stream);
    mlbm_status st = mlbm_lattice_step(L, n_steps);
    cudaEventRecord(e1, L->stream);
    cudaError_t e = cudaEventSynchronize(e1);
    float t = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&t, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st != MLBM_OK) return st;
    if (e != cudaSuccess) return set_error(MLBM_E_CUDA, std::string("lattice_time_steps: ") + cudaGetErrorString(e));
    *ms = t;
    return MLBM_OK;
}

mlbm_status mlbm_lattice_sync(mlbm_lattice* L) {
    if (!L) return set_error(MLBM_E_INVALID, "lattice_sync: NULL lattice");
    LAT_CUDA(cudaStreamSynchronize(L->stream));
    return MLBM_OK;
}

mlbm_status mlbm_lattice_set_populations(mlbm_lattice* L, const double* f) {
    if (!L || !f) return set_error(MLBM_E_INVALID, "lattice_set_populations: NULL argument");
    const size_t n = (size_t)L->nx * L->ny;
    LAT_CUDA(cudaMemcpyAsync(L->io, f, 9 * n * sizeof(double), cudaMemcpyHostToDevice, L->stream));
    dev::lattice_set<<<(unsigned)((n + 255) / 256), 256, 0, L->stream>>>(n, L->io, L->f[L->cur]);
    LAT_CUDA(cudaGetLastError());
    LAT_CUDA(cudaStreamSynchronize(L->stream));
    L->steps = 0;
    return MLBM_OK;
}

mlbm_status mlbm_lattice_get_populations(mlbm_lattice* L, double* f) {
    if (!L || !f) return set_error(MLBM_E_INVALID, "lattice_get_populations: NULL argument");
    const size_t n = (size_t)L->nx * L->ny;
    dev::lattice_get<<<(unsigned)((n + 255) / 256), 256, 0, L->stream>>>(n, L->f[L->cur], L->io);
    LAT_CUDA(cudaGetLastError());
    LAT_CUDA(cudaMemcpyAsync(f, L->io, 9 * n * sizeof(double), cudaMemcpyDeviceToHost, L->stream));
    LAT_CUDA(cudaStreamSynchronize(L->stream));
    return MLBM_OK;
}

mlbm_status mlbm_lattice_force(mlbm_lattice* L, double* fx, double* fy) {
    if (!L) return set_error(MLBM_E_INVALID, "lattice_force: NULL lattice");
    dev::lattice_force<<<1, 256, 0, L->stream>>>((size_t)L->nx * L->ny, L->n_wall, L->wall, L->f[L->cur], L->small);
    LAT_CUDA(cudaGetLastError());
    double h[2];
    LAT_CUDA(cudaMemcpyAsync(h, L->small, 16, cudaMemcpyDeviceToHost, L->stream));
    LAT_CUDA(cudaStreamSynchronize(L->stream));
    if (fx) *fx = h[0];
    if (fy) *fy = h[1];
    return MLBM_OK;
}

}  // extern "C"
