// Backward Monte Carlo with the sun local estimate (Eq. ble): paths start at a camera, fly
// through the staged extinction grid by the voxel walk of the forward transport, and at every
// scattering event add the sun's single-scattered radiance toward the camera. The paper uses it
// to check the in-situ forward model (Sec. 3); here it renders whole images, a path at a time
// per thread, every pixel on its own Philox stream (counter word 3 = 1 + global pixel index).
#include <algorithm>
#include <cmath>

#include "mst_internal.h"

namespace mst {
namespace {

constexpr int kTB = 256;

__device__ __forceinline__ bool inside(const Geo& g, int ix, int iy, int iz) {
    return (unsigned)ix < (unsigned)g.nx && (unsigned)iy < (unsigned)g.ny && (unsigned)iz < (unsigned)g.nz;
}

struct BmcArgs {
    Geo g;
    CamSet cams;
    HG hg;
    const void* beta;       // staged extinction on the padded grid (halo +inf)
    const float* omega;     // [total pix] pixel solid angles
    float3 to_sun;          // unit vector toward the sun
    float albedo, F;        // single-scattering albedo, sun irradiance
    float rr_below, rr_survival, inv_rr_survival;
    uint2 key;
    int max_order, max_events;
    uint32_t n;             // paths per pixel
    uint64_t total;         // total pixels x n
    double* sum;            // [total pix] sum of path values
    double* sum2;           // [total pix] sum of squared path values
    double* stats;          // [MST_NSTATS]
};

// offset along one axis of the point a distance l past the walk's current point (d: the direction
// component, p0: the walk's start); the multiply-add is spelled out, so that a path does not depend
// on what the compiler fuses around it
__device__ __forceinline__ float bmc_offset(float t, float d, float h, float p0, float l) {
    const float v = d > 0.f ? fmaf(-(t - l), d, h) : (d < 0.f ? __fmul_rn(t - l, -d) : p0);
    return fminf(fmaxf(v, 0.f), h);
}

// One path: its pixel and number, the point it stands at (voxel + offset) and its direction, the free path
// drawn for the next flight, its weight, the events so far and what the sun has given it.
struct Path {
    uint32_t gp, q, ev;
    float3 p, d;
    int ix, iy, iz;
    float tau, I;
    double wpix, contrib;
};

// path t begins at its pixel; false when its ray misses the grid
__device__ __forceinline__ bool path_start(const BmcArgs& A, uint64_t t, Path& s) {
    s.gp = (uint32_t)(t / A.n);
    s.q = (uint32_t)(t - (uint64_t)s.gp * A.n);
    const int c = cam_of_pixel(A.cams, (int)s.gp);
    const Cam& cm = A.cams.c[c];
    const int li = (int)s.gp - cm.pix_off, i = li % cm.w, j = li / cm.w;
    const float4 u = draws(A.key, s.q, 0u, 1u + s.gp);
    const float px = (float)i + u.x, py = (float)j + u.y;
    const float xx = (2.f * px / (float)cm.w - 1.f) * cm.tx, yy = (2.f * py / (float)cm.h - 1.f) * cm.ty;
    const float cosv = rsqrtf(1.f + xx * xx + yy * yy);
    const float apix = (2.f * cm.tx / (float)cm.w) * (2.f * cm.ty / (float)cm.h);
    s.wpix = (double)(cosv * cosv * cosv) * (double)apix / (double)A.omega[s.gp];
    s.d = pixel_dir(cm, px, py);
    s.contrib = 0.0;
    s.I = 1.f;
    s.tau = -logf(1.f - u.z);
    s.ev = 0u;
    return ray_start(A.g, cm, s.d, s.p, s.ix, s.iy, s.iz);
}

// the flight ended a distance l into the walk's voxel (jx, jy, jz): the path stands there
__device__ __forceinline__ void path_collide(const BmcArgs& A, Path& s, const PadWalk& w, float l, int jx, int jy, int jz) {
    ++s.ev;
    s.p = make_float3(bmc_offset(w.tx, s.d.x, A.g.hx, s.p.x, l), bmc_offset(w.ty, s.d.y, A.g.hy, s.p.y, l),
                      bmc_offset(w.tz, s.d.z, A.g.hz, s.p.z, l));
    s.ix = jx;
    s.iy = jy;
    s.iz = jz;
}

// the sun's local estimate of the event (its ray left through the top face)
__device__ __forceinline__ void path_sunlit(const BmcArgs& A, Path& s, const PairSum& depth) {
    const float mu = s.d.x * A.to_sun.x + s.d.y * A.to_sun.y + s.d.z * A.to_sun.z;
    s.contrib += (double)(A.albedo * s.I * hg_phase(A.hg, mu)) * exp(-depth.value()) * (double)A.F;
}

// on from the event: albedo, order and event limits, roulette, the new direction and free path
__device__ __forceinline__ bool path_scatter(const BmcArgs& A, Path& s) {
    s.I *= A.albedo;
    if (s.I == 0.f || (A.max_order > 0 && (int)s.ev >= A.max_order) || (int)s.ev >= A.max_events) return false;
    const float4 u = draws(A.key, s.q, s.ev, 1u + s.gp);
    if (s.I < A.rr_below) {
        if (!(u.z < A.rr_survival)) return false;
        s.I *= A.inv_rr_survival;
    }
    float ct, st;
    hg_sample(A.hg, u.x, ct, st);
    s.d = rotate_dir(s.d, ct, st, u.y);
    s.tau = -logf(1.f - u.w);
    return true;
}

__device__ __forceinline__ void path_finish(const BmcArgs& A, const Path& s) {
    const double v = s.contrib * s.wpix;
    if (v != 0.0) {
        atomicAdd(A.sum + s.gp, v);
        atomicAdd(A.sum2 + s.gp, v * v);
    }
}

__device__ __forceinline__ void flush_counts(const BmcArgs& A, unsigned paths, unsigned events, unsigned nseg) {
    const unsigned long long np = warp_sumu(paths), ne = warp_sumu(events), ns = warp_sumu(nseg);
    if ((threadIdx.x & 31u) == 0u) {
        atomicAdd(A.stats + MST_ST_BMC_PATHS, (double)np);
        atomicAdd(A.stats + MST_ST_BMC_EVENTS, (double)ne);
        atomicAdd(A.stats + MST_ST_BMC_SEGMENTS, (double)ns);
    }
}

// A lane walks one ray at a time, a path's free flight or the sun-ward ray of its event, by the
// same voxel step on the padded grid, kBmcTrip voxels at a time; between trips the lanes whose ray
// has ended do what follows it (the collision, the event, the next path). Lanes stay busy whatever
// their rays' lengths: 64 paths a pixel of 9 cameras of 128^2 pixels in 64^3 voxels take 17.1 ms, 19.3 with
// the rays walked to their ends in turn (k_bmc_small).
// Trips of 24 / 32 / 48 voxels ran 5.7 / 5.7 / 5.9 ms with three blocks an SM (16 paths a pixel), 32 ran
// 5.0 with four (64 registers).
constexpr int kBmcTrip = 32;
constexpr int kBmcBlocks = 4;  // per SM

template <int DT>
__global__ void __launch_bounds__(kTB, kBmcBlocks) k_bmc(const BmcArgs A) {
    unsigned paths = 0u, events = 0u, nseg = 0u;
    const uint64_t stride = (uint64_t)gridDim.x * kTB;
    uint64_t t = (uint64_t)blockIdx.x * kTB + threadIdx.x;  // the lane's next path
    enum { kIdle, kFlight, kSun } ray = kIdle;
    PadWalk w{};
    float bn = 0.f;  // extinction of the walk's voxel, loaded one step ahead
    int left = 0;    // voxel steps before a walk is abandoned (only a non-finite direction gets there)
    PairSum depth;   // sun ray: optical depth so far
    Path s{};
    auto start = [&](bool sun) {
        w = pad_walk(A.g, s.p, sun ? A.to_sun : s.d, s.ix, s.iy, s.iz);
        bn = BetaFetch<DT>::get(A.beta, w.lin);
        left = A.g.max_steps;
        depth = PairSum();
        ray = sun ? kSun : kFlight;
    };
    for (;;) {
        while (ray == kIdle && t < A.total) {  // the next path that enters the grid
            ++paths;
            if (path_start(A, t, s)) start(false);
            t += stride;
        }
        if (!__any_sync(0xffffffffu, ray != kIdle)) break;
        // up to kBmcTrip voxels
        bool end = false;
        float b = 0.f;
        if (ray != kIdle) {
            const bool sun = ray == kSun;
#pragma unroll 1
            for (int n = 0; n < kBmcTrip; ++n) {
                b = bn;
                bool px, py;
                int next;
                const float m = w.face(px, py, next);
                bn = BetaFetch<DT>::get(A.beta, next);  // at most the second halo layer
                const float bs = __fmul_rn(b, m);
                if (ray_ends(!sun, s.tau, b, bs)) {
                    end = true;
                    break;
                }
                ++nseg;
                if (sun) depth.add(bs);
                else s.tau -= bs;
                w.cross(m, px, py, next);
            }
            left -= kBmcTrip;
        }
        bool done = false;
        if (end) {
            int jx, jy, jz;
            unpad(A.g, w.lin, jx, jy, jz);
            const bool in = inside(A.g, jx, jy, jz);
            if (ray == kFlight) {
                done = !in || isnan(b);  // (no path collides in a voxel without an extinction)
                if (!done) {  // a collision: the sun's local estimate
                    ++nseg;
                    ++events;
                    path_collide(A, s, w, s.tau / b, jx, jy, jz);
                    start(true);
                }
            } else {  // (an infinite extinction inside the grid: nothing of the sun arrives)
                if (!in && jz >= A.g.nz) path_sunlit(A, s, depth);
                left = -1;
            }
        }
        if (ray != kIdle && left < 0 && !done) {
            if (!end) atomicAdd(A.stats + MST_ST_LOST, 1.0);  // abandoned
            if (ray == kSun && path_scatter(A, s)) start(false);
            else done = true;
        }
        if (done) {
            path_finish(A, s);
            ray = kIdle;
        }
    }
    flush_counts(A, paths, events, nseg);
}

// The same paths, each lane walking a flight, the sun ray of its event and the next flight to their ends
// in turn, the lanes of a warp coming together after each walk (__syncwarp): the event's FP64 and
// Philox rounds then run once for them, not once for every length that a walk had (without: 64 x 64
// x 2 voxels 0.46 ms against 0.29, 16^3 0.94 against 0.67).
// It takes grids with an extent below kBmcSmall voxels, whose walks differ too little for k_bmc's trips
// (ms here / there: 1 x 256 x 256 0.90 / 1.36, 8^3 1.0 / 1.9, 16^3 0.70 / 1.19, 32^3 3.2 / 3.6, 48^3 8.6 / 8.9,
// 96^3 11.9 / 10.8), and calls with fewer than kBmcPerLane paths for each resident lane, which k_bmc
// ends on its lanes' last paths (64^3 at 3.8 paths a lane 1.6 / 1.9, at 7.6 2.96 / 3.05, at 15 5.3 / 5.0, at 61
// 19.3 / 17.1).
constexpr int kBmcSmall = 64;
constexpr int kBmcPerLane = 10;
template <int DT>
__global__ void __launch_bounds__(kTB, kBmcBlocks) k_bmc_small(const BmcArgs A) {
    unsigned paths = 0u, events = 0u, nseg = 0u;
    const uint64_t stride = (uint64_t)gridDim.x * kTB;
    for (uint64_t t = (uint64_t)blockIdx.x * kTB + threadIdx.x; t < A.total; t += stride) {
        Path s;
        ++paths;
        if (!path_start(A, t, s)) continue;
        PadWalk w;
        PairSum depth;
        float b = 0.f;
        int jx, jy, jz;
        // to the ray's end; false when it was abandoned
        auto walk = [&](bool sun) {
            const unsigned together = __activemask();  // every one of them reaches the __syncwarp
            w = pad_walk(A.g, s.p, sun ? A.to_sun : s.d, s.ix, s.iy, s.iz);
            float bn = BetaFetch<DT>::get(A.beta, w.lin);
            depth = PairSum();
            int n = 0;
#pragma unroll 1
            for (; n <= A.g.max_steps; ++n) {
                b = bn;
                bool px, py;
                int next;
                const float m = w.face(px, py, next);
                bn = BetaFetch<DT>::get(A.beta, next);  // at most the second halo layer
                const float bs = __fmul_rn(b, m);
                if (ray_ends(!sun, s.tau, b, bs)) break;
                ++nseg;
                if (sun) depth.add(bs);
                else s.tau -= bs;
                w.cross(m, px, py, next);
            }
            __syncwarp(together);
            if (n > A.g.max_steps) {
                atomicAdd(A.stats + MST_ST_LOST, 1.0);
                return false;
            }
            unpad(A.g, w.lin, jx, jy, jz);
            return true;
        };
        while (walk(false) && inside(A.g, jx, jy, jz) && !isnan(b)) {
            ++nseg;
            ++events;
            path_collide(A, s, w, s.tau / b, jx, jy, jz);
            if (walk(true) && !inside(A.g, jx, jy, jz) && jz >= A.g.nz) path_sunlit(A, s, depth);
            if (!path_scatter(A, s)) break;
        }
        path_finish(A, s);
    }
    flush_counts(A, paths, events, nseg);
}

// Pixel means and the variance of each mean from the path sums.
__global__ void k_bmc_finish(double* __restrict__ mean, double* __restrict__ sum2, double* __restrict__ var,
                             int npix, uint32_t n) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < npix; k += gridDim.x * blockDim.x) {
        const double m = mean[k] / n;
        mean[k] = m;
        if (var) var[k] = n > 1 ? (sum2[k] / n - m * m) / (double)(n - 1) : 0.0;
    }
}

}  // namespace

cudaError_t launch_bmc(const mst_grid* g, const mst_params* p, uint32_t n, double* sum, double* sum2, double* var,
                       cudaStream_t st) {
    BmcArgs a;
    a.g = g->geo;
    a.cams = g->cams;
    const double gg = p->g;
    a.hg.g = (float)gg;
    a.hg.k1 = (float)((1.0 - gg * gg) / (4.0 * M_PI));
    a.hg.a = (float)(1.0 + gg * gg);
    a.hg.b = (float)(2.0 * gg);
    a.hg.omg2 = (float)(1.0 - gg * gg);
    a.hg.omg = (float)(1.0 - gg);
    a.hg.opg = (float)(1.0 + gg);
    a.hg.tg = (float)(2.0 * gg);
    a.hg.iso = std::fabs(gg) < 1e-6;
    a.beta = g->ext_pad;
    a.omega = g->omega;
    const double th = p->sun_zenith_rad, ph = p->sun_azimuth_rad;
    a.to_sun = make_float3((float)(std::sin(th) * std::cos(ph)), (float)(std::sin(th) * std::sin(ph)), (float)std::cos(th));
    a.albedo = (float)p->albedo;
    a.F = (float)p->sun_irradiance;
    a.rr_below = (float)p->rr_threshold;
    a.rr_survival = (float)p->rr_survival;
    a.inv_rr_survival = (float)(1.0 / p->rr_survival);
    a.key = make_uint2((uint32_t)p->seed, (uint32_t)(p->seed >> 32));
    a.max_order = p->max_order;
    a.max_events = p->max_events;
    a.n = n;
    a.total = (uint64_t)g->total_pix * n;
    a.sum = sum;
    a.sum2 = sum2;
    a.stats = g->stats;
    const uint64_t lanes = (uint64_t)g->sm_count * kBmcBlocks * kTB;
    const bool small = std::min(std::min(g->geo.nx, g->geo.ny), g->geo.nz) < kBmcSmall || a.total < kBmcPerLane * lanes;
    auto go = [&](auto machine, auto in_turn) {
        // k_bmc's blocks are resident at once: a lane takes its paths one after another
        if (small) in_turn<<<g->sm_count * 8, kTB, 0, st>>>(a);
        else machine<<<g->sm_count * kBmcBlocks, kTB, 0, st>>>(a);
    };
    if (p->grid_dtype == 0) go(k_bmc<0>, k_bmc_small<0>);
    else if (p->grid_dtype == 1) go(k_bmc<1>, k_bmc_small<1>);
    else go(k_bmc<2>, k_bmc_small<2>);
    const int nb = (g->total_pix + kTB - 1) / kTB;
    k_bmc_finish<<<nb < 4096 ? nb : 4096, kTB, 0, st>>>(sum, sum2, var, g->total_pix, n);
    return cudaGetLastError();
}

}  // namespace mst
