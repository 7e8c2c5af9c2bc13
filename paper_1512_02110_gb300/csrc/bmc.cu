// Backward Monte Carlo with the sun local estimate (Eq. ble): paths start at a camera, fly
// through the staged extinction grid by the voxel walk of the forward transport, and at every
// scattering event add the sun's single-scattered radiance toward the camera. The paper uses it
// to check the in-situ forward model (Sec. 3); here it renders whole images, one path per
// thread, every pixel on its own Philox stream (counter word 3 = 1 + global pixel index).
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

// A lane walks one ray at a time, a path's free flight or the sun-ward ray of its event, by the
// same voxel step on the padded grid, kBmcTrip voxels at a time; between trips the lanes whose ray
// has ended do what follows it (the collision, the event, the next path). Lanes stay busy whatever
// their rays' lengths: walking flight and sun ray to their ends in turn, each lane waiting for the
// longest of its warp, took 7.5 ms against 4.9 for 2.4e6 paths (64^3, 9 cameras of 128^2 pixels), and 10.6
// ms with voxel indices, bounds tests and FP64 depths in every step.
// Trips of 24 / 32 / 48 voxels ran 5.7 / 5.7 / 5.9 ms with three blocks an SM, 32 ran 4.9 with four
// (64 registers).
constexpr int kBmcTrip = 32;
constexpr int kBmcBlocks = 4;  // per SM

template <int DT>
__global__ void __launch_bounds__(kTB, kBmcBlocks) k_bmc(const BmcArgs A) {
    unsigned paths = 0u, events = 0u, nseg = 0u;
    const uint64_t stride = (uint64_t)gridDim.x * kTB;
    uint64_t t = (uint64_t)blockIdx.x * kTB + threadIdx.x;  // the lane's next path
    enum { kIdle, kFlight, kSun } ray = kIdle;
    PadWalk w{};
    float bn = 0.f;       // extinction of the walk's voxel, loaded one step ahead
    int left = 0;         // voxel steps before a walk is abandoned (only a non-finite direction gets there)
    float tau = 0.f;      // flight: free path left
    PairSum depth;        // sun ray: optical depth so far
    float3 p = make_float3(0.f, 0.f, 0.f), d = p;
    int ix = 0, iy = 0, iz = 0;
    uint32_t gp = 0u, q = 0u, ev = 0u;
    float I = 0.f;
    double wpix = 0.0, contrib = 0.0;
    auto start = [&](bool sun) {
        w = pad_walk(A.g, p, sun ? A.to_sun : d, ix, iy, iz);
        bn = BetaFetch<DT>::get(A.beta, w.lin);
        left = A.g.max_steps;
        depth = PairSum();
        ray = sun ? kSun : kFlight;
    };
    auto finish = [&]() {  // the path is done
        const double v = contrib * wpix;
        if (v != 0.0) {
            atomicAdd(A.sum + gp, v);
            atomicAdd(A.sum2 + gp, v * v);
        }
        ray = kIdle;
    };
    for (;;) {
        while (ray == kIdle && t < A.total) {  // the next path that enters the grid
            gp = (uint32_t)(t / A.n);
            q = (uint32_t)(t - (uint64_t)gp * A.n);
            t += stride;
            const int c = cam_of_pixel(A.cams, (int)gp);
            const Cam& cm = A.cams.c[c];
            const int li = (int)gp - cm.pix_off, i = li % cm.w, j = li / cm.w;
            const float4 u = draws(A.key, q, 0u, 1u + gp);
            const float px = (float)i + u.x, py = (float)j + u.y;
            const float xx = (2.f * px / (float)cm.w - 1.f) * cm.tx, yy = (2.f * py / (float)cm.h - 1.f) * cm.ty;
            const float cosv = rsqrtf(1.f + xx * xx + yy * yy);
            const float apix = (2.f * cm.tx / (float)cm.w) * (2.f * cm.ty / (float)cm.h);
            wpix = (double)(cosv * cosv * cosv) * (double)apix / (double)A.omega[gp];
            d = pixel_dir(cm, px, py);
            contrib = 0.0;
            ++paths;
            if (ray_start(A.g, cm, d, p, ix, iy, iz)) {
                I = 1.f;
                tau = -logf(1.f - u.z);
                ev = 0u;
                start(false);
            }
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
                if (ray_ends(!sun, tau, b, bs)) {
                    end = true;
                    break;
                }
                ++nseg;
                if (sun) depth.add(bs);
                else tau -= bs;
                w.cross(m, px, py, next);
            }
            left -= kBmcTrip;
        }
        if (end) {
            int jx, jy, jz;
            unpad(A.g, w.lin, jx, jy, jz);
            const bool in = inside(A.g, jx, jy, jz);
            if (ray == kFlight) {
                if (!in) {
                    finish();
                } else {  // a collision: the sun's local estimate
                    ++nseg;
                    ++events;
                    ++ev;
                    const float l = tau / b;
                    p = make_float3(bmc_offset(w.tx, d.x, A.g.hx, p.x, l), bmc_offset(w.ty, d.y, A.g.hy, p.y, l),
                                    bmc_offset(w.tz, d.z, A.g.hz, p.z, l));
                    ix = jx;
                    iy = jy;
                    iz = jz;
                    start(true);
                }
            } else if (in) {  // an infinite extinction inside the grid: nothing of the sun arrives
                left = -1;
            } else {
                if (jz >= A.g.nz) {  // the sun-ward ray leaves through the top face: sunlit
                    const float mu = d.x * A.to_sun.x + d.y * A.to_sun.y + d.z * A.to_sun.z;
                    contrib += (double)(A.albedo * I * hg_phase(A.hg, mu)) * exp(-depth.value()) * (double)A.F;
                }
                left = -1;
            }
        }
        if (ray != kIdle && left < 0) {
            if (!end) atomicAdd(A.stats + MST_ST_LOST, 1.0);  // abandoned
            if (ray == kFlight) {
                finish();
            } else {  // on from the event
                I *= A.albedo;
                bool on = I != 0.f && !(A.max_order > 0 && (int)ev >= A.max_order) && (int)ev < A.max_events;
                if (on) {
                    const float4 u = draws(A.key, q, ev, 1u + gp);
                    if (I < A.rr_below) {
                        if (u.z < A.rr_survival) I *= A.inv_rr_survival;
                        else on = false;
                    }
                    if (on) {
                        float ct, st;
                        hg_sample(A.hg, u.x, ct, st);
                        d = rotate_dir(d, ct, st, u.y);
                        tau = -logf(1.f - u.w);
                        start(false);
                    }
                }
                if (!on) finish();
            }
        }
    }
    const unsigned long long np = warp_sumu(paths), ne = warp_sumu(events), ns = warp_sumu(nseg);
    if ((threadIdx.x & 31u) == 0u) {
        atomicAdd(A.stats + MST_ST_BMC_PATHS, (double)np);
        atomicAdd(A.stats + MST_ST_BMC_EVENTS, (double)ne);
        atomicAdd(A.stats + MST_ST_BMC_SEGMENTS, (double)ns);
    }
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
    const int blocks = g->sm_count * kBmcBlocks;  // resident at once: a lane takes its paths one after another
    if (p->grid_dtype == 0) k_bmc<0><<<blocks, kTB, 0, st>>>(a);
    else if (p->grid_dtype == 1) k_bmc<1><<<blocks, kTB, 0, st>>>(a);
    else k_bmc<2><<<blocks, kTB, 0, st>>>(a);
    const int nb = (g->total_pix + kTB - 1) / kTB;
    k_bmc_finish<<<nb < 4096 ? nb : 4096, kTB, 0, st>>>(sum, sum2, var, g->total_pix, n);
    return cudaGetLastError();
}

}  // namespace mst
