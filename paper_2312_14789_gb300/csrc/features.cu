// Geometry features of the learned warm start (one thread per node; positions
// as pairs of floats, FP32 geometry)
// and the kernels that turn a network prediction into an initial state.
//
// Features (16 per node, L = length scale, ell = min(8 L, min(Lx, Ly) / 2)):
//   0      clamp(d1 / L, 0, 4), d1 = distance to the nearest solid surface
//   1, 2   unit vector from that surface point to the node
//   3      clamp(d2 / L, 0, 4), d2 = distance to the second nearest solid object
//   4..7   free paths along +x, -x, +y, -y: distance to the first solid along
//          the ray, at most ell, over L
//   8      clamp(f(+y) f(-y) / L^2, 0, 16)  (the cross-stream Poiseuille
//          profile y (w - y) of a channel along x)
//   9      clamp((f(+y) + f(-y)) / L, 0, 8) (cross-stream gap width)
//   10..13 local porosity within radius rho_j = min(c_j L, min(Lx, Ly) / 2),
//          c_j = 1, 2, 4, 8: 1 - (solid area in the circle) / (pi rho_j^2),
//          disks and their periodic images as circle-circle lenses, solid
//          sides as circular segments
//   14     porosity of the box
//   15     4 (y - y0) (y1 - y) / Ly^2 (position across the box)
// Objects are visited in a fixed order (disks in input order, periodic
// images ix = -1, 0, 1 outer and iy inner around the minimum image, then the
// solid sides left, right, bottom, top); the first strictly nearer object
// sets the direction.  A ray meets a disk when its entry point lies at
// t >= -1e-4 r (a node on the surface looking into the disk sees it at 0,
// looking outward it sees no hit).
#include <cmath>
#include <string>
#include <vector>

#include "kernels.h"
#include "mlbm_internal.h"

namespace mlbm {
namespace dev {

constexpr double kPi = 3.141592653589793238462643383279502884;
constexpr float kPif = 3.14159265358979f;

// area of the intersection of two circles of radii a and b, centres d apart:
// two circular segments cut by the common chord.  The chord's half-length
// comes from the product form of Heron's formula and the segment angles from
// atan2 of (half-chord, signed centre-to-chord distance), which stays well
// conditioned in FP32 near tangency and near containment (acos of a cosine
// near +-1 does not).
__device__ float lens_area(float d, float a, float b) {
    if (d >= a + b) return 0.f;
    if (d <= fabsf(a - b)) {
        const float m = fminf(a, b);
        return kPif * m * m;
    }
    const float k = fmaxf(0.f, (-d + a + b) * (d + a - b) * (d - a + b) * (d + a + b));
    const float hc = sqrtf(k) / (2.f * d);
    const float xa = (d * d + a * a - b * b) / (2.f * d);  // signed distance from centre A to the chord
    const float xb = d - xa;
    return a * a * atan2f(hc, xa) - xa * hc + b * b * atan2f(hc, xb) - xb * hc;
}

// area of the part of a circle of radius a beyond a line at signed distance h
// from its centre (half-angle from atan2 for the same reason)
__device__ float segment_area(float h, float a) {
    if (h >= a) return 0.f;
    if (h <= -a) return kPif * a * a;
    const float hc = sqrtf((a - h) * (a + h));
    return a * a * atan2f(hc, h) - h * hc;
}

constexpr int kRadii = 4;

struct FeatGeo {
    double x0, y0, lx, ly;
    int perx, pery;
    int solid[4];
    int n_disks;
    float L, ell;
    float rho[kRadii];
    float porosity;
};

// entry distance of a ray along +a (sign = +1) or -a (sign = -1) into a disk,
// da = node - centre along the ray axis, db across it (|db| <= r); the
// half-chord is formed as a product of sums, which keeps its accuracy at
// grazing incidence; INFINITY when the entry lies behind the start (by more
// than 1e-4 r, which absorbs the rounding of a start on the surface)
__device__ __forceinline__ float ray_entry(float da, float db, float r, float sign) {
    const float adb = fabsf(db);
    const float t = -sign * da - sqrtf((r - adb) * (r + adb));
    return t >= -1e-4f * r ? fmaxf(t, 0.f) : INFINITY;
}

// a - b with the error of the FP32 subtraction (Knuth's TwoSum)
__device__ __forceinline__ void diff2(float a, float b, float& s, float& e) {
    s = __fsub_rn(a, b);
    const float bb = __fsub_rn(a, s);
    e = __fadd_rn(__fsub_rn(a, __fadd_rn(s, bb)), __fsub_rn(bb, b));
}

// A double as two floats (48 bits): positions and disk centres from the box's
// corner (taken off in FP64, so that a box far from the origin keeps its bits),
// and box lengths.  Differences of them are formed with their rounding errors,
// which gives the FP32 displacement to its last bit or so; in FP64 the subtraction, the
// division by the box length and the conversions of every disk were most of
// the kernel on this GPU (two FP64 instructions per clock and SM).
struct Two {
    float h, l;
};
__device__ __forceinline__ Two two_of(double x) {
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}
// minimum image of x - c along an axis of length L (periodic when per != 0)
__device__ __forceinline__ float image_diff(const Two& x, const Two& c, const Two& L, int per) {
    float s, e;
    diff2(x.h, c.h, s, e);
    e += x.l - c.l;
    if (per) {
        const float m = rintf((s + e) / L.h);
        if (m != 0.f) {
            float p = __fmul_rn(m, L.h);  // m is a small integer
            const float pe = __fmaf_rn(m, L.h, -p);
            float s2, e2;
            diff2(s, p, s2, e2);
            s = s2;
            e += e2 - pe - m * L.l;
        }
    }
    return s + e;
}

struct Disk {
    Two x, y;
    float r;
    float bx, by;  // centre from the box's corner, moved into the box along periodic axes
};

// Disks that can come within `reach` of a point of each grid cell (any of
// their periodic images), in disk order: one block per cell, list[cell * cap
// ..], count[cell], cells and centres counted from the box's corner.  margin
// covers FP32 rounding.
__global__ void __launch_bounds__(128) bin_disks(FeatGeo G, const Disk* __restrict__ disks, int ncx, int ncy,
                                                 float cw, float ch, float reach, int* __restrict__ list,
                                                 int* __restrict__ count) {
    __shared__ int warp_n[4], base;
    const int cx = blockIdx.x % ncx, cy = blockIdx.x / ncx;
    const float x0 = cx * cw, y0 = cy * ch, x1 = x0 + cw, y1 = y0 + ch;
    const float lx = (float)G.lx, ly = (float)G.ly;
    const float margin = 1e-4f * (reach + lx + ly);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int* out = list + (size_t)blockIdx.x * G.n_disks;
    if (threadIdx.x == 0) base = 0;
    __syncthreads();
    for (int k0 = 0; k0 < G.n_disks; k0 += 128) {
        const int k = k0 + threadIdx.x;
        bool near = false;
        if (k < G.n_disks) {
            const Disk d = disks[k];
            const float lim = reach + d.r + margin + 1e-6f * (fabsf(d.bx) + fabsf(d.by) + fabsf(d.r));
            for (int ix = -2 * G.perx; ix <= 2 * G.perx; ++ix)
                for (int iy = -2 * G.pery; iy <= 2 * G.pery; ++iy) {
                    const float X = d.bx + ix * lx, Y = d.by + iy * ly;
                    const float dx = fmaxf(0.f, fmaxf(x0 - X, X - x1)), dy = fmaxf(0.f, fmaxf(y0 - Y, Y - y1));
                    near |= dx * dx + dy * dy <= lim * lim;
                }
        }
        const unsigned vote = __ballot_sync(0xffffffffu, near);
        if (lane == 0) warp_n[warp] = __popc(vote);
        __syncthreads();
        int at = base;
        for (int w = 0; w < warp; ++w) at += warp_n[w];
        if (near) out[at + __popc(vote & ((1u << lane) - 1u))] = k;
        __syncthreads();
        if (threadIdx.x == 0) base += warp_n[0] + warp_n[1] + warp_n[2] + warp_n[3];
        __syncthreads();
    }
    if (threadIdx.x == 0) count[blockIdx.x] = base;
}

// One thread per node over the disks listed for its cell, in disk order, so
// every sum and every choice is the one over all disks: a disk that is not
// listed is at least `reach` away, where it cuts no circle and no ray, and it
// can only matter as one of the two nearest objects when fewer than two listed
// ones are closer; such nodes look again at all disks.  Bound by the lens
// areas of the ~45 listed disks of a node (two arc tangents each where a disk
// cuts one of the four circles).  192k nodes, 212 disks: 1310 us with every
// disk and image in FP64, 150 us now.
__global__ void __launch_bounds__(128) features_kernel(int64_t n, const double* __restrict__ xy,
                                                       const Disk* __restrict__ disks, FeatGeo G, int ncx, int ncy,
                                                       float cw, float ch, const int* __restrict__ list,
                                                       const int* __restrict__ count, float* __restrict__ X) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = xy[2 * i], y = xy[2 * i + 1];
    const Two x2 = two_of(x - G.x0), y2 = two_of(y - G.y0), lx2 = two_of(G.lx), ly2 = two_of(G.ly);
    float d1 = INFINITY, d2 = INFINITY, nx = 0.f, ny = 0.f;
    float fp[4] = {G.ell, G.ell, G.ell, G.ell};  // +x, -x, +y, -y
    float S[kRadii] = {0.f, 0.f, 0.f, 0.f};
    auto take = [&](float d, float ux, float uy) {
        if (d < d1) {
            d2 = d1;
            d1 = d;
            nx = ux;
            ny = uy;
        } else if (d < d2) {
            d2 = d;
        }
    };
    const float reach = fmaxf(G.rho[kRadii - 1], G.ell);  // beyond it a disk cuts no circle and no ray
    const float lxf = (float)G.lx, lyf = (float)G.ly;
    // the node's cell (a node outside the box takes all disks)
    const float px = x2.h, py = y2.h;
    const bool inside = ncx > 0 && px >= 0.f && py >= 0.f && px <= lxf && py <= lyf;
    const int cell = inside ? min(ncy - 1, (int)(py / ch)) * ncx + min(ncx - 1, (int)(px / cw)) : 0;
    const int* ids = inside ? list + (size_t)cell * G.n_disks : nullptr;
    const int m = inside ? count[cell] : G.n_disks;
    for (int q = 0; q < m; ++q) {
        const Disk D = disks[ids ? ids[q] : q];
        const float r = D.r;
        const float dx0 = image_diff(x2, D.x, lx2, G.perx), dy0 = image_diff(y2, D.y, ly2, G.pery);
        for (int ix = -G.perx; ix <= G.perx; ++ix)
            for (int iy = -G.pery; iy <= G.pery; ++iy) {
                const float dx = dx0 + ix * lxf, dy = dy0 + iy * lyf;
                const float dist = sqrtf(dx * dx + dy * dy);
                const float d = dist - r;
                if (d < d2) {
                    if (d < d1) take(d, dist > 0.f ? dx / dist : 0.f, dist > 0.f ? dy / dist : 0.f);
                    else d2 = d;
                }
                if (d >= reach) continue;
                if (fabsf(dy) <= r) {
                    fp[0] = fminf(fp[0], ray_entry(dx, dy, r, 1.f));
                    fp[1] = fminf(fp[1], ray_entry(dx, dy, r, -1.f));
                }
                if (fabsf(dx) <= r) {
                    fp[2] = fminf(fp[2], ray_entry(dy, dx, r, 1.f));
                    fp[3] = fminf(fp[3], ray_entry(dy, dx, r, -1.f));
                }
#pragma unroll
                for (int j = 0; j < kRadii; ++j) S[j] += lens_area(dist, G.rho[j], r);
            }
    }
    if (inside && !(d2 < reach) && m < G.n_disks) {  // fewer than two objects near: the nearest of all
        d1 = d2 = INFINITY;
        nx = ny = 0.f;
        for (int k = 0; k < G.n_disks; ++k) {
            const Disk D = disks[k];
            const float dx0 = image_diff(x2, D.x, lx2, G.perx), dy0 = image_diff(y2, D.y, ly2, G.pery);
            for (int ix = -G.perx; ix <= G.perx; ++ix)
                for (int iy = -G.pery; iy <= G.pery; ++iy) {
                    const float dx = dx0 + ix * lxf, dy = dy0 + iy * lyf;
                    const float dist = sqrtf(dx * dx + dy * dy);
                    take(dist - D.r, dist > 0.f ? dx / dist : 0.f, dist > 0.f ? dy / dist : 0.f);
                }
        }
    }
    const float h[4] = {(float)(x - G.x0), (float)(G.x0 + G.lx - x), (float)(y - G.y0), (float)(G.y0 + G.ly - y)};
    const float wn[4][2] = {{1, 0}, {-1, 0}, {0, 1}, {0, -1}};
    const int ray_of_side[4] = {1, 0, 3, 2};  // the -x ray meets the left side, ...
#pragma unroll
    for (int sd = 0; sd < 4; ++sd) {
        if (!G.solid[sd]) continue;
        take(h[sd], wn[sd][0], wn[sd][1]);
        fp[ray_of_side[sd]] = fminf(fp[ray_of_side[sd]], fmaxf(h[sd], 0.f));
#pragma unroll
        for (int j = 0; j < kRadii; ++j) S[j] += segment_area(h[sd], G.rho[j]);
    }
    if (!(d1 < INFINITY)) d1 = 4.f * G.L;
    if (!(d2 < INFINITY)) d2 = 4.f * G.L;
    const float a = d1 / G.L, b = d2 / G.L;
    float* o = X + 16 * i;
    o[0] = fminf(fmaxf(a, 0.f), 4.f);
    o[1] = nx;
    o[2] = ny;
    o[3] = fminf(fmaxf(b, 0.f), 4.f);
#pragma unroll
    for (int j = 0; j < 4; ++j) o[4 + j] = fp[j] / G.L;
    o[8] = fminf(fp[2] * fp[3] / (G.L * G.L), 16.f);
    o[9] = fminf((fp[2] + fp[3]) / G.L, 8.f);
#pragma unroll
    for (int j = 0; j < kRadii; ++j) o[10 + j] = 1.f - S[j] / (kPif * G.rho[j] * G.rho[j]);
    o[14] = G.porosity;
    const double yy = y - G.y0;
    o[15] = (float)(4.0 * yy * (G.ly - yy) / (G.ly * G.ly));
}

// ---------------------------------------------------------------- warm start
// Y[n][no] (caller order): scaled velocity in columns 0, 1 and, when no = 3,
// scaled density deviation in column 2.
// flag[sample] |= 1 when a prediction of the sample is unusable: a
// non-finite value, a speed above umax or a density deviation above drho_max
__global__ void warm_check(int n, const int* __restrict__ perm, const uint16_t* __restrict__ node_sample,
                           const uint8_t* __restrict__ meta, const float* __restrict__ Y, int no,
                           const double* __restrict__ scale_u, const double* __restrict__ scale_rho, float umax,
                           float drho_max, int* __restrict__ flag) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    if ((meta[p] & 3) == 2) return;  // equilibrium-overwrite node
    const int smp = node_sample ? node_sample[p] : 0;
    const int64_t id = perm[p];
    const double ux = scale_u[smp] * (double)Y[no * id], uy = scale_u[smp] * (double)Y[no * id + 1];
    const double sp = sqrt(ux * ux + uy * uy);
    bool bad = !(sp <= (double)umax);
    if (no == 3) bad |= !(fabs(scale_rho[smp] * (double)Y[no * id + 2]) <= (double)drho_max);
    if (bad) atomicOr(&flag[smp], 1);
}

// scaled density deviation of every node in position order (0 on
// equilibrium-overwrite nodes), for the per-sample mean
__global__ void warm_drho(int n, const int* __restrict__ perm, const uint16_t* __restrict__ node_sample,
                          const uint8_t* __restrict__ meta, const float* __restrict__ Y, int no,
                          const double* __restrict__ scale_rho, float* __restrict__ drho) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int smp = node_sample ? node_sample[p] : 0;
    drho[p] = (meta[p] & 3) == 2 ? 0.f : (float)(scale_rho[smp] * (double)Y[no * (int64_t)perm[p] + 2]);
}

// area-weighted mean of drho over every sample's masked nodes (0 without any):
// partial sums of A and drho A per block, then one block per sample
__global__ void __launch_bounds__(256) warm_means_partial(const int64_t* __restrict__ seg, int max_nb,
                                                          const float* __restrict__ drho,
                                                          const float* __restrict__ area,
                                                          const uint8_t* __restrict__ mask,
                                                          double* __restrict__ partial) {
    const int64_t first = seg[blockIdx.y], end = seg[blockIdx.y + 1];
    double a = 0.0, d = 0.0;
    for (int64_t i = first + blockIdx.x * 256LL + threadIdx.x; i < end; i += (int64_t)max_nb * 256)
        if (mask[i]) {
            a += area[i];
            d += (double)drho[i] * area[i];
        }
    __shared__ double sa[256], sd[256];
    sa[threadIdx.x] = a;
    sd[threadIdx.x] = d;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) {
            sa[threadIdx.x] += sa[threadIdx.x + h];
            sd[threadIdx.x] += sd[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        partial[2 * ((size_t)blockIdx.y * max_nb + blockIdx.x)] = sa[0];
        partial[2 * ((size_t)blockIdx.y * max_nb + blockIdx.x) + 1] = sd[0];
    }
}
__global__ void __launch_bounds__(32) warm_means_final(int max_nb, const double* __restrict__ partial,
                                                       double* __restrict__ mean) {
    double a = 0.0, d = 0.0;
    for (int b = threadIdx.x; b < max_nb; b += 32) {
        a += partial[2 * ((size_t)blockIdx.x * max_nb + b)];
        d += partial[2 * ((size_t)blockIdx.x * max_nb + b) + 1];
    }
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        d += __shfl_xor_sync(0xffffffffu, d, o);
    }
    if (threadIdx.x == 0) mean[blockIdx.x] = a > 0.0 ? d / a : 0.0;
}

// rho_u[n][3] (caller order, FP64) of the warm start: rho = 1 + (predicted
// deviation - its area-weighted sample mean, so the sample's mass stays that
// of the rest state) and u = predicted velocity; samples flagged cold start
// from rest; equilibrium-overwrite nodes take their boundary values
__global__ void warm_fill(int n, const int* __restrict__ perm, const uint16_t* __restrict__ node_sample,
                          const uint8_t* __restrict__ meta, const float4* __restrict__ eqv,
                          const float* __restrict__ Y, int no, const double* __restrict__ scale_u,
                          const float* __restrict__ drho, const double* __restrict__ drho_mean,
                          const int* __restrict__ flag, double* __restrict__ ru) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int smp = node_sample ? node_sample[p] : 0;
    const int64_t id = perm[p];
    double* v = ru + 3 * id;
    if ((meta[p] & 3) == 2) {
        const float4 e = eqv[p];
        v[0] = 1.0 + (double)e.x;
        v[1] = e.y;
        v[2] = e.z;
        return;
    }
    const bool cold = flag[smp] != 0;
    const double sc = cold ? 0.0 : scale_u[smp];
    v[0] = (no == 3 && !cold) ? 1.0 + ((double)drho[p] - drho_mean[smp]) : 1.0;
    v[1] = sc * (double)Y[no * id];
    v[2] = sc * (double)Y[no * id + 1];
}

}  // namespace dev

cudaError_t launch_warm_check(int n, const int* perm, const uint16_t* node_sample, const uint8_t* meta,
                              const float* Y, int no, const double* scale_u, const double* scale_rho, float umax,
                              float drho_max, int* flag, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    dev::warm_check<<<(n + 255) / 256, 256, 0, st>>>(n, perm, node_sample, meta, Y, no, scale_u, scale_rho, umax,
                                                     drho_max, flag);
    return cudaGetLastError();
}

cudaError_t launch_warm_drho(int n, const int* perm, const uint16_t* node_sample, const uint8_t* meta,
                             const float* Y, int no, const double* scale_rho, float* drho, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    dev::warm_drho<<<(n + 255) / 256, 256, 0, st>>>(n, perm, node_sample, meta, Y, no, scale_rho, drho);
    return cudaGetLastError();
}

cudaError_t launch_warm_means(int ns, int max_nb, const int64_t* seg, const float* drho, const float* area,
                              const uint8_t* mask, double* partial, double* mean, cudaStream_t st) {
    dev::warm_means_partial<<<dim3(max_nb, ns), 256, 0, st>>>(seg, max_nb, drho, area, mask, partial);
    dev::warm_means_final<<<ns, 32, 0, st>>>(max_nb, partial, mean);
    return cudaGetLastError();
}

cudaError_t launch_warm_fill(int n, const int* perm, const uint16_t* node_sample, const uint8_t* meta,
                             const float4* eqv, const float* Y, int no, const double* scale_u, const float* drho,
                             const double* drho_mean, const int* flag, double* ru, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    dev::warm_fill<<<(n + 255) / 256, 256, 0, st>>>(n, perm, node_sample, meta, eqv, Y, no, scale_u, drho, drho_mean,
                                                    flag, ru);
    return cudaGetLastError();
}

}  // namespace mlbm

using namespace mlbm;

extern "C" mlbm_status mlbm_features_device(const mlbm_nodes* nodes, const mlbm_geometry* geo, double L, float* X) {
    clear_error();
    if (!nodes || !geo || !X || nodes->n < 0 || (nodes->n > 0 && !nodes->xy) || !(L > 0) ||
        (geo->n_disks > 0 && !geo->disks) || geo->n_disks < 0)
        return set_error(MLBM_E_INVALID, "features: bad arguments");
    const double lx = geo->x1 - geo->x0, ly = geo->y1 - geo->y0;
    if (!(lx > 0) || !(ly > 0)) return set_error(MLBM_E_INVALID, "features: empty box");
    const int64_t n = nodes->n;
    if (n == 0) return MLBM_OK;
    dev::FeatGeo G{};
    G.x0 = geo->x0;
    G.y0 = geo->y0;
    G.lx = lx;
    G.ly = ly;
    G.perx = geo->side[0] == MLBM_SIDE_PERIODIC && geo->side[1] == MLBM_SIDE_PERIODIC;
    G.pery = geo->side[2] == MLBM_SIDE_PERIODIC && geo->side[3] == MLBM_SIDE_PERIODIC;
    for (int k = 0; k < 4; ++k) G.solid[k] = geo->side[k] == MLBM_SIDE_SOLID;
    G.n_disks = geo->n_disks;
    G.L = (float)L;
    G.ell = (float)std::fmin(8.0 * L, 0.5 * std::fmin(lx, ly));
    const double cj[dev::kRadii] = {1.0, 2.0, 4.0, 8.0};
    for (int j = 0; j < dev::kRadii; ++j) G.rho[j] = (float)std::fmin(cj[j] * L, 0.5 * std::fmin(lx, ly));
    double solid = 0.0;
    for (int k = 0; k < geo->n_disks; ++k) solid += dev::kPi * geo->disks[3 * k + 2] * geo->disks[3 * k + 2];
    G.porosity = (float)(1.0 - solid / (lx * ly));
    // grid of the disk lists: cells of a quarter of the reach, at most 32 MB
    // of lists (fewer, longer cells in a thin box), none when the disks are few
    // enough to look at all of them
    const int nd = geo->n_disks;
    const double reach = std::fmax((double)G.rho[dev::kRadii - 1], (double)G.ell);
    int ncx = 0, ncy = 0;
    if (nd >= 16) {
        const double most = std::fmax(1.0, std::floor(double(32 << 20) / sizeof(int) / nd));  // cells
        const double edge = std::fmax(0.25 * reach, std::sqrt(lx * ly / most));
        const double wide = std::ceil(lx / edge), high = std::ceil(ly / edge);
        ncx = (int)std::fmax(1.0, std::fmin(wide, most / std::fmin(high, most)));
        ncy = (int)std::fmax(1.0, std::fmin(high, most / ncx));
    }
    const size_t cells = (size_t)ncx * ncy;
    std::vector<dev::Disk> hd(nd);
    auto two = [](double v) {
        const float h = (float)v;
        return dev::Two{h, (float)(v - (double)h)};
    };
    for (int k = 0; k < nd; ++k) {
        const double cx = geo->disks[3 * k] - G.x0, cy = geo->disks[3 * k + 1] - G.y0;  // from the box's corner
        hd[k] = {two(cx), two(cy), (float)geo->disks[3 * k + 2],
                 (float)(G.perx ? cx - lx * std::floor(cx / lx) : cx),
                 (float)(G.pery ? cy - ly * std::floor(cy / ly) : cy)};
    }
    // one buffer: positions, disks, lists, counts
    const size_t bytes_xy = (size_t)n * 2 * sizeof(double), bytes_d = ((size_t)nd * sizeof(dev::Disk) + 15) / 16 * 16;
    uint8_t* buf = nullptr;
    cudaError_t e = cudaMalloc(&buf, bytes_xy + bytes_d + cells * ((size_t)nd + 1) * sizeof(int));
    if (e == cudaSuccess) {
        double* dxy = reinterpret_cast<double*>(buf);
        dev::Disk* dd = reinterpret_cast<dev::Disk*>(buf + bytes_xy);
        int* count = reinterpret_cast<int*>(buf + bytes_xy + bytes_d);
        int* list = count + cells;
        const float cw = cells ? (float)(lx / ncx) : 1.f, ch = cells ? (float)(ly / ncy) : 1.f;
        if (nd > 0) e = cudaMemcpyAsync(dd, hd.data(), nd * sizeof(dev::Disk), cudaMemcpyHostToDevice, nullptr);
        if (e == cudaSuccess && cells)
            dev::bin_disks<<<(unsigned)cells, 128>>>(G, dd, ncx, ncy, cw, ch, (float)reach, list, count);
        if (e == cudaSuccess) e = cudaMemcpyAsync(dxy, nodes->xy, bytes_xy, cudaMemcpyHostToDevice, nullptr);
        if (e == cudaSuccess) {
            dev::features_kernel<<<(unsigned)((n + 127) / 128), 128>>>(n, dxy, dd, G, ncx, ncy, cw, ch, list, count, X);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
    }
    cudaFree(buf);
    if (e != cudaSuccess) return set_error(MLBM_E_CUDA, std::string("features: ") + cudaGetErrorString(e));
    return MLBM_OK;
}
