// Host-side launchers of the kernels in kernels.cu.
#pragma once

#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>
#include <vector>

#include "device_common.cuh"

namespace mlbm {

cudaError_t launch_bgk_step(const dev::Stencil& S, const float4* f8in, const float* f0in, float4* f8out,
                            float* f0out, const dev::Collide& C, int variant, cudaStream_t st);
// wall tractions of the listed wall nodes (device positions pos[m], normals
// nrm[m][2], wall lengths ds[m]) into out[m][2], FP64 (wall_stress.cu)
cudaError_t launch_wall_traction(const dev::Stencil& S, int model, const float4* f8, const float* f0,
                                 const float4* ruv, float ax, float ay, double nu, double s, const int* pos,
                                 const double* nrm, const double* ds, int m, double* out, cudaStream_t st);
// raises the dynamic shared-memory limit of the staged step kernel (variant 22)
cudaError_t prepare_staged_step(int Kq, int stage_max);
// BGK variants 0-3 (kernels_bgk_generic.cu)
cudaError_t launch_bgk_step_generic(const dev::Stencil& S, const float4* f8in, const float* f0in, float4* f8out,
                                    float* f0out, const dev::Collide& C, int variant, cudaStream_t st);
// BGK variants 14-19 and 22 (kernels_bgk_alt.cu)
cudaError_t launch_bgk_step_alt(const dev::Stencil& S, const float4* f8in, const float* f0in, float4* f8out,
                                float* f0out, const dev::Collide& C, int variant, cudaStream_t st);
// RBF-FD stencils (kernels_rbf.cu); launch_bgk_step / launch_tau1_step hand
// contexts with per-direction weights to these
cudaError_t launch_bgk_step_rbf(const dev::Stencil& S, const float4* f8in, const float* f0in, float4* f8out,
                                float* f0out, const dev::Collide& C, int variant, cudaStream_t st);
cudaError_t launch_tau1_step_rbf(const dev::Stencil& S, const float4* in, float4* out, const dev::Collide& C,
                                 int variant, cudaStream_t st);
cudaError_t launch_tau1_step(const dev::Stencil& S, const float4* in, float4* out, const dev::Collide& C, int variant,
                             cudaStream_t st);
cudaError_t launch_set_bgk(int n, const int* perm, const double* f, float4* f8, float* f0, cudaStream_t st);
cudaError_t launch_get_bgk(int n, const int* perm, const float4* f8, const float* f0, double* f, cudaStream_t st);
cudaError_t launch_set_bgk_equilibrium(int n, const int* perm, const double* ru, float4* f8, float* f0,
                                       cudaStream_t st);
cudaError_t launch_set_tau1(int n, const int* perm, const double* ru, float4* s, cudaStream_t st);
// tau = 1: holds the m nodes' states fixed in later steps by making them
// equilibrium-kind nodes whose record is their current state (run to steady
// state of a batch: samples that have converged)
cudaError_t launch_freeze_tau1(int first, int m, uint8_t* meta, float4* eqv, const float4* state, cudaStream_t st);
// brings the tile records and what each tile fetches in line with the kind
// bytes after they changed; no step may be launched before the stream has
// been synchronised
cudaError_t launch_record_kinds(const dev::Stencil& S, float4* rec, uint8_t* need, int* range, cudaStream_t st);
// blocks (and tile ranges) of the per-warp-slot step for n nodes
int warp_step_ranges(int n);
// one step of every partition (variants 27..29): the partitions' ranges in one
// launch, new halo states stored straight into the receivers' slots
cudaError_t launch_step_parts(int model, int Kq, int64_t n, const dev::PartDev* parts, const int2* work, int blocks,
                              int from, int* err, const dev::Wait& W, cudaStream_t st);
cudaError_t launch_mark_sends(int n, const int* send_first, uint8_t* meta, cudaStream_t st);
// halo slots of all partitions from their owners' states in buffer `cur`, w
// float4 a state
cudaError_t launch_exchange(const dev::PartDev* parts, const int4* list, int64_t m, int w, int cur, cudaStream_t st);
// step kernels with a shared-memory slot per warp (kernels_warp.cu), variants
// 27..29; backward walks the tiles from the last one where that is of use
cudaError_t launch_step_warp(int variant, int model, const dev::Stencil& S, const float4* a8, const float* a0,
                             float4* b8, float* b0, const float4* ra, float4* rb, const dev::Collide& C, int backward,
                             int* err, const dev::Wait& W, cudaStream_t st);
// many BGK steps of a small set by one cluster that keeps everything in shared
// memory (kernels_cluster.cu): its size for a set (0: does not fit), and
// `steps` steps from one state into another (the same buffers, or others)
int step_cluster_size(int Kq, int n);
cudaError_t launch_step_cluster(int size, const dev::Stencil& S, const float4* in, const float* f0in, float4* out,
                                float* f0out, const dev::Collide& C, int steps, int* err, const dev::Wait& W,
                                cudaStream_t st);
// RBF-FD tile records (kernels_rbf_tiles.cu; tiles of 16 nodes): their sizes,
// the layout from the sizes (false where they do not fit), their contents,
// and the step from them
cudaError_t rbf_tile_sizes(const dev::Stencil& S, int tiles, int2* size, cudaStream_t st);
bool rbf_tiles_plan(const std::vector<int2>& size, int blocks, std::vector<int4>& head, std::vector<int>& range,
                    int& slot, size_t& bytes);
cudaError_t rbf_tile_fill(const dev::Stencil& S, int tiles, const int4* head, uint8_t* rec, cudaStream_t st);
cudaError_t launch_step_rbf_tiles(const dev::Stencil& S, const float4* in, const float* f0in, float4* out,
                                  float* f0out, const dev::Collide& C, int backward, int* err, const dev::Wait& W,
                                  cudaStream_t st);
cudaError_t launch_macroscopics(int model, int n, const int* perm, const float4* f8, const float* f0,
                                const float4* ruv, float ax, float ay, const uint16_t* node_sample,
                                const dev::Collide* coll, int split, double* out, cudaStream_t st);
// persistent bulk-copy pipelined step (kernels_tma.cu), variants 4..7
bool tma_supported(int Kq);
cudaError_t launch_step_tma(int variant, int model, const dev::Stencil& S, const float4* f8in, const float* f0in,
                            float4* f8out, float* f0out, const float4* rin, float4* rout, const dev::Collide& C,
                            int* err, const dev::Wait& W, cudaStream_t st);
int force_blocks(int n_link_nodes);
cudaError_t launch_force(const dev::Stencil& S, int model, int n_link_nodes, const int* link_nodes,
                         const float* area_over_s2, const float4* f8, const float4* ruv, const dev::Collide& C,
                         double* partial, double* out, cudaStream_t st);
// the FP64 reductions never use more than this many partial-sum blocks
constexpr int kReduceMaxBlocks = 1024;
int reduce_blocks(int64_t n);
cudaError_t launch_reduce_fields(const float* rho, const float* ux, const float* uy, const float* area,
                                 const uint8_t* mask, int64_t n, double* partial, double* out, cudaStream_t st);
// observables of all samples of a context from its state, `out` [sample][W]:
// kObserveChange (W = 3) sum |u - u_prev|^2, sum |u|^2 and the count of nodes
// with a non-positive density or non-finite field, then u -> u_prev (px, py);
// kObserveFields (W = 6) the sums of launch_reduce_fields; kObserveBoth (W =
// 9).  seg (device): first position of each sample and the end; max_nb:
// reduce_blocks of the largest sample; partial: ns * max_nb * W doubles
enum { kObserveChange = 3, kObserveFields = 6, kObserveBoth = 9 };
cudaError_t launch_observe(int model, int what, int ns, int max_nb, const int64_t* seg, const float4* f8,
                           const float* f0, const float4* ruv, const dev::Collide& C, const dev::Collide* coll,
                           const float* area, const uint8_t* mask, float* px, float* py, double* partial, double* out,
                           cudaStream_t st);

// warm start (features.cu)
cudaError_t launch_warm_check(int n, const int* perm, const uint16_t* node_sample, const uint8_t* meta,
                              const float* Y, int no, const double* scale_u, const double* scale_rho, float umax,
                              float drho_max, int* flag, cudaStream_t st);
cudaError_t launch_warm_drho(int n, const int* perm, const uint16_t* node_sample, const uint8_t* meta,
                             const float* Y, int no, const double* scale_rho, float* drho, cudaStream_t st);
// area-weighted mean of drho per sample (0 where the areas sum to nothing);
// partial: 2 * ns * max_nb doubles
cudaError_t launch_warm_means(int ns, int max_nb, const int64_t* seg, const float* drho, const float* area,
                              const uint8_t* mask, double* partial, double* mean, cudaStream_t st);
cudaError_t launch_warm_fill(int n, const int* perm, const uint16_t* node_sample, const uint8_t* meta,
                             const float4* eqv, const float* Y, int no, const double* scale_u, const float* drho,
                             const double* drho_mean, const int* flag, double* ru, cudaStream_t st);

}  // namespace mlbm
