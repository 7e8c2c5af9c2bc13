// Deterministic ray kernels of the voxelised model: grid staging, LOS transmittance
// (Eq. taoKtoc-Tck), pixel-ray image formation (Eq. Icpixel) with the loss epilogue
// (Eq. Cost), back-projection Pi^T, the LOS adjoint W^T, sub-pixel ray counts (Sec. 6),
// the gradient combinations of Eq. Jaco1-DivTc and the Laplacian regulariser.
//
// Geometry is never stored: every Pi_c and W_c product re-walks its rays through the grid.
// LOS threads run x-fastest over voxels of one camera, so a warp walks 32 nearly parallel
// rays toward the same X_c.
#include <cmath>

#include "mst_internal.h"

namespace mst {
namespace {

constexpr int kTB = 256;
constexpr int kRayBlock = 256;  // threads of a pixel-ray block (n_rays <= 64 divide it into whole pixels)

// threads of a block that hold a ray: the largest multiple of n_rays within kRayBlock
__host__ __device__ __forceinline__ int pixel_rays_block(int n_rays) { return kRayBlock / n_rays * n_rays; }

// The extinction in FP32 in the linear voxel order of the input, for the call without a handle.
__global__ void k_stage(const float* __restrict__ beta, float* __restrict__ ext, int nvox) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nvox; k += gridDim.x * blockDim.x) ext[k] = beta[k];
}

// The grid that every ray and flight walks: the extinction in the compute dtype on
// [nz + 4][ny + 4][nx + 4] with a halo of +inf, where a walk stops (a free path never outlasts
// infinite optical depth). Two species (Sec. 2): beta = beta_aerosol + beta_air, and the FP32 total
// for the surrogate's j = L / beta.
template <int DT>
__global__ void k_stage_pad(const float* __restrict__ beta, const float* __restrict__ air, void* __restrict__ ext,
                            float* __restrict__ tot, const Geo g) {
    typedef typename BetaFetch<DT>::T T;
    T* out = static_cast<T*>(ext);
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < g.npad; q += gridDim.x * blockDim.x) {
        const int ix = q % g.p0 - kHalo, iy = (q / g.p0) % (g.ny + 2 * kHalo) - kHalo, iz = q / g.p01 - kHalo;
        float b = CUDART_INF_F;
        if (ix >= 0 && ix < g.nx && iy >= 0 && iy < g.ny && iz >= 0 && iz < g.nz) {
            const int k = lin_index(g, ix, iy, iz);
            b = air ? beta[k] + air[k] : beta[k];
            if (tot) tot[k] = b;
        }
        out[q] = BetaFetch<DT>::make(b);
    }
}

// beta_ref + beta_air in FP32 (the surrogate's reference total)
__global__ void k_add_air(const float* __restrict__ beta, const float* __restrict__ air, float* __restrict__ out,
                          int nvox) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nvox; k += gridDim.x * blockDim.x) out[k] = beta[k] + air[k];
}

// Adds the block's segment count to its statistic: one FP64 atomic per block (one per warp put
// 8.6e5 of them on one address at 768e3 voxels x 36 cameras). Called by every thread of the block.
__device__ __forceinline__ void block_count(double* stats, int slot, unsigned n) {
    __shared__ unsigned total;
    if (threadIdx.x == 0) total = 0u;
    __syncthreads();
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31u) == 0u && n) atomicAdd(&total, n);
    __syncthreads();
    if (threadIdx.x == 0 && total) atomicAdd(stats + slot, (double)total);
}

// R is stored on the padded grid with this bit pattern in its halo, which no arithmetic produces
// (a computed NaN is 0x7FFFFFFF): a pixel ray that loads it has left the grid.
constexpr int kOutside = -1;

// length from the current point (the walk stands in the camera's voxel) to the centre of projection
__device__ __forceinline__ float camera_leg(const Geo& g, const Cam& c, const PadWalk& w, float3 d, float3 p) {
    // spelled out, so that no other choice of fused multiply-adds moves T by an ulp
    auto local = [](float t, float dd, float h, float p0) {
        const float v = dd > 0.f ? __fsub_rn(h, __fmul_rn(t, dd)) : (dd < 0.f ? __fmul_rn(t, -dd) : p0);
        return fminf(fmaxf(v, 0.f), h);
    };
    const float3 q = make_float3(local(w.tx, d.x, g.hx, p.x), local(w.ty, d.y, g.hy, p.y), local(w.tz, d.z, g.hz, p.z));
    return fmaf(__fsub_rn(c.lz, q.z), d.z, fmaf(__fsub_rn(c.lx, q.x), d.x, __fmul_rn(__fsub_rn(c.ly, q.y), d.y)));
}

// direction from the centre of voxel (ix, iy, iz) to camera c and the distance; false at the centre itself
__device__ __forceinline__ bool los_dir(const Geo& g, const Cam& c, int ix, int iy, int iz, float3& p, float3& d,
                                        float& dist) {
    p = make_float3(0.5f * g.hx, 0.5f * g.hy, 0.5f * g.hz);
    const float3 v = local_delta(g, ix, iy, iz, p, c.ix, c.iy, c.iz, make_float3(c.lx, c.ly, c.lz));
    dist = sqrtf(v.x * v.x + v.y * v.y + v.z * v.z);
    if (!(dist > 0.f)) return false;
    const float inv = 1.f / dist;
    d = make_float3(v.x * inv, v.y * inv, v.z * inv);
    return true;
}

// K2: tau_c(k) along the LOS from the centre of voxel k to X_c; T = exp(-tau). With L given,
// also R_c(k) = L_c(k) T_c(k) (Eq. Rck) on the padded grid, where L = Lsrc * beta / beta_ref when
// beta_ref is given (the j-fixed surrogate, L = j beta with j = L_ref / beta_ref). The walk ends in
// the camera's voxel, at the grid's boundary (the first halo voxel) or when the distance is used up.
// PAD: the field is on the padded grid and its halo (+inf) ends the walk, the next voxel loaded one
// step ahead. Without a padded copy (the call that allocates nothing) the walk counts the voxels
// left to the boundary on each axis instead.
template <int DT, bool PAD>
__global__ void __launch_bounds__(kTB) k_los(const Geo g, const CamSet cs, const void* __restrict__ ext,
                                             const double* __restrict__ Lsrc, const float* __restrict__ beta_ref,
                                             const float* __restrict__ beta, float* __restrict__ T_out,
                                             float* __restrict__ R_out, double* stats) {
    const int c = blockIdx.y, k = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned nseg = 0u;
    if (k < g.nvox) {
        const Cam& cm = cs.c[c];
        const size_t idx = (size_t)c * g.nvox + k;
        const int ix = k % g.nx, iy = (k / g.nx) % g.ny, iz = k / (g.nx * g.ny);
        PairSum tau;
        float3 p, d;
        float rem;
        if (los_dir(g, cm, ix, iy, iz, p, d, rem)) {
            const int goal = !cm.inside ? -1 : (PAD ? pad_index(g, cm.ix, cm.iy, cm.iz) : lin_index(g, cm.ix, cm.iy, cm.iz));
            PadWalk w(g, p, d, PAD ? pad_index(g, ix, iy, iz) : k, PAD ? g.p0 : g.nx, PAD ? g.p01 : g.nx * g.ny);
            FacesLeft left(g, d, ix, iy, iz);
            float b, m, bn = BetaFetch<DT>::get(ext, w.lin);
            bool px, py;
            int next;
            for (;;) {  // one exit, whatever ends the walk: the loop is bound by its instructions
                b = bn;
                m = w.face(px, py, next);
                if (PAD) bn = BetaFetch<DT>::get(ext, next);  // the walk stands inside: next is at most in the halo
                if ((PAD && isinf(b)) || w.lin == goal || m >= rem || nseg >= (unsigned)g.max_steps) break;
                ++nseg;
                tau.add(__fmul_rn(b, m));
                rem -= m;
                if (!PAD && left.out(px, py)) {
                    m = -1.f;
                    break;
                }
                w.cross(m, px, py, next);
                if (!PAD) bn = BetaFetch<DT>::get(ext, w.lin);
            }
            int q;
            if (m >= 0.f && (!PAD || !isinf(b) || interior_lin(g, w.lin, q))) {  // not in the halo: the last voxel
                ++nseg;
                if (w.lin == goal) m = fmaxf(camera_leg(g, cm, w, d, p), 0.f);
                tau.add(__fmul_rn(b, fminf(m, rem)));
            }
        }
        const float T = (float)exp(-tau.value());
        if (T_out) T_out[idx] = T;
        if (R_out) {
            double L = Lsrc[idx];
            if (beta_ref) {
                const float br = beta_ref[k];
                L = br > 0.f ? L * (double)beta[k] / (double)br : 0.0;
            }
            R_out[(size_t)c * g.npad + pad_index(g, ix, iy, iz)] = (float)(L * (double)T);
        }
    }
    if (stats) block_count(stats, MST_ST_LOS_SEGMENTS, nseg);
}

// The pixel rays of a block: thread t takes sub-pixel ray t % n_rays of pixel first + t / n_rays, so
// a warp's rays belong to two to four neighbouring pixels (10 rays each) and cross the same
// voxels for most of their way.
struct PixelRay {
    int pixels, gp, rho;  // pixels of a block, this thread's pixel and ray
    bool on;
    __device__ __forceinline__ PixelRay(int n_rays, int total_pix) {
        pixels = pixel_rays_block(n_rays) / n_rays;
        const int q = threadIdx.x / n_rays;
        rho = threadIdx.x - q * n_rays;
        gp = blockIdx.x * pixels + q;
        on = q < pixels && gp < total_pix;
    }
};

// start of pixel gp's ray rho; false when it misses the grid
__device__ __forceinline__ bool pixel_ray_start(const Geo& g, const Cam& cm, const Halton& hs, int gp, int rho, float3& p,
                                                float3& d, int& ix, int& iy, int& iz) {
    const int q = gp - cm.pix_off, i = q % cm.w, j = q / cm.w;
    d = pixel_dir(cm, (float)i + hs.a[rho], (float)j + hs.b[rho]);
    return ray_start(g, cm, d, p, ix, iy, iz);
}

// K3: i_c(p) = 1/(N_rays V) sum_rho sum_k l(k) R_c(k) (Eq. Icpixel). With measurements, also
// r = M (i - i_meas), resid = 2 r = dE/di, and E += r^2 (Eq. Cost). One thread per ray; the pixel's
// rays are added in FP64 in their order. A thread per pixel walked its rays one after another:
// 0.61 ms against 0.15 at 9 cameras of 128^2 pixels in 64^3 voxels, 59 against 15 us at 5 cameras
// of 32^2 pixels in 16^3, where the call waited for ten walks in a row.
__global__ void k_images(const Geo g, const CamSet cs, const Halton hs, float inv_nv, const float* __restrict__ R,
                         double* __restrict__ images, const double* __restrict__ meas, const uint8_t* __restrict__ mask,
                         double* __restrict__ resid, double* loss, int total_pix, double* stats) {
    __shared__ double part[kRayBlock];
    const PixelRay ray(hs.n, total_pix);
    unsigned nseg = 0u;
    PairSum acc;
    if (ray.on) {
        const int c = cam_of_pixel(cs, ray.gp);
        const Cam& cm = cs.c[c];
        float3 p, d;
        int ix, iy, iz;
        if (pixel_ray_start(g, cm, hs, ray.gp, ray.rho, p, d, ix, iy, iz)) {
            const float* Rc = R + (size_t)c * g.npad;
            PadWalk w = pad_walk(g, p, d, ix, iy, iz);
            float rn = __ldg(Rc + w.lin);
            for (;;) {
                const float r = rn;
                if (__float_as_int(r) == kOutside) break;
                ++nseg;
                bool px, py;
                int next;
                const float m = w.face(px, py, next);
                rn = __ldg(Rc + next);
                acc.add(__fmul_rn(m, r));
                if (nseg > (unsigned)g.max_steps) break;
                w.cross(m, px, py, next);
            }
        }
    }
    part[threadIdx.x] = acc.value();
    __syncthreads();
    if (threadIdx.x < 32) {
        double r2 = 0.0;
        for (int q = threadIdx.x; q < ray.pixels; q += 32) {
            const int gp = blockIdx.x * ray.pixels + q;
            if (gp >= total_pix) break;
            double s = 0.0;
            for (int rho = 0; rho < hs.n; ++rho) s += part[q * hs.n + rho];
            const double img = s * (double)inv_nv;
            if (images) images[gp] = img;
            if (meas) {
                const double r = (mask && !mask[gp]) ? 0.0 : img - meas[gp];
                resid[gp] = 2.0 * r;
                r2 += r * r;
            }
        }
        if (meas) {
            r2 = warp_sum(r2);
            if (threadIdx.x == 0 && r2 != 0.0) atomicAdd(loss, r2);
        }
    }
    if (stats) block_count(stats, MST_ST_PIXEL_SEGMENTS, nseg);
}

// K4: b_c(k) = sum_p Pi_c(p, k) resid(p)  (Pi^T, Eq. PIc transposed). A thread takes a pixel and walks
// its rays in their order, counting the faces left to the boundary (stopping on the halo mark of R
// instead, a load per voxel, took 1.37 ms for the 36 cameras of 64^2 pixels over 80 x 80 x 120 voxels
// against 1.30, and 76 us for 3 cameras of 8^2 pixels over 96^3 against 21). An atomic on an address that
// another lane of the instruction holds costs another transaction (2.0e11 a second on this chip,
// however many lanes share it); what bounds the kernel is the queue on each camera's own voxel (1.6e5
// additions). 9 cameras of 128^2 pixels in 64^3 voxels: 0.86-0.95 ms. A warp taking every fourth pixel,
// whose rays part sooner, took 0.85, and adding the lanes' terms up before the atomic 0.27; neither was
// kept: the bins next to a camera sum so many terms in FP32 that another order moves them by up to 1e-3.
// Below this many pixels a camera, the rays of a pixel go to threads of their own: few pixels leave the
// chip to single threads' chains of rays (us apart / in one thread, by pixels a camera: 64: 15 / 82 (1 camera, 64^3),
// 9 / 35 (5, 16^3); 576: 31 / 123, 23 / 37). They are faster apart up to some 3000 pixels (2025: 64 / 135, 56 / 60;
// 4096: 127 / 160, 146 / 109), but from 32^2 on the order of the FP32 sums decides: apart, the bins next to a
// camera move by two to five times what two runs of one form differ by.
constexpr int kRaysApart = 1024;
__global__ void __launch_bounds__(kTB) k_backproject(const Geo g, const CamSet cs, const Halton hs, float inv_nv,
                                                     const double* __restrict__ resid, float* __restrict__ bacc,
                                                     int total_pix, double* stats) {
    const int gp = blockIdx.x * kTB + (int)threadIdx.x;
    unsigned nseg = 0u;
    const float wgt = gp < total_pix ? (float)(resid[gp] * (double)inv_nv) : 0.f;
    if (wgt != 0.f) {
        const int c = cam_of_pixel(cs, gp);
        float* bc = bacc + (size_t)c * g.nvox;
        for (int rho = blockIdx.y; rho < hs.n; rho += gridDim.y) {
            float3 p, d;
            int ix, iy, iz;
            if (!pixel_ray_start(g, cs.c[c], hs, gp, rho, p, d, ix, iy, iz)) continue;
            PadWalk w(g, p, d, lin_index(g, ix, iy, iz), g.nx, g.nx * g.ny);
            FacesLeft left(g, d, ix, iy, iz);
            for (int n = 0; n <= g.max_steps; ++n) {
                ++nseg;
                bool px, py;
                int next;
                const float m = w.face(px, py, next);
                if (m > 0.f) atomicAdd(bc + w.lin, wgt * m);
                if (left.out(px, py)) break;
                w.cross(m, px, py, next);
            }
        }
    }
    if (stats) block_count(stats, MST_ST_BACKPROJ_SEGMENTS, nseg);
}

// K5: gT_c(m) = sum_k W_c(k, m) s_c(k), s = R b = L T b (Eq. DivTc transposed).
// Every line of a camera ends in its voxel, where the atomics queue up on one address. With more voxels
// than the chip has threads at once the blocks therefore go round the cameras (TURN), so that the
// queues run side by side (36 cameras over 80 x 80 x 120 voxels: 12.1 ms camera after camera, 3.3 ms
// in turn). On smaller grids the lines of several cameras are under way anyway (64^3, 9 cameras: 0.13
// against 0.10 ms), and camera after camera keeps the order in which a bin's FP32 terms arrive.
template <bool TURN>
__global__ void __launch_bounds__(kTB) k_los_adjoint(const Geo g, const CamSet cs, const float* __restrict__ R,
                                                     const float* __restrict__ bacc, float* __restrict__ gT,
                                                     double* stats) {
    const int nb = gridDim.x / cs.n;  // blocks of a camera
    const int c = TURN ? blockIdx.x % cs.n : blockIdx.x / nb;
    const int k = (int)(TURN ? blockIdx.x / cs.n : blockIdx.x % nb) * kTB + (int)threadIdx.x;
    unsigned nseg = 0u;
    if (k < g.nvox) {
        const Cam& cm = cs.c[c];
        float* gc = gT + (size_t)c * g.nvox;
        const int ix = k % g.nx, iy = (k / g.nx) % g.ny, iz = k / (g.nx * g.ny);
        const float s = R[(size_t)c * g.npad + pad_index(g, ix, iy, iz)] * bacc[(size_t)c * g.nvox + k];
        float3 p, d;
        float rem;
        if (s != 0.f && los_dir(g, cm, ix, iy, iz, p, d, rem)) {
            const int goal = cm.inside ? lin_index(g, cm.ix, cm.iy, cm.iz) : -1;
            PadWalk w(g, p, d, k, g.nx, g.nx * g.ny);
            FacesLeft left(g, d, ix, iy, iz);
            float m;
            bool px, py;
            int next;
            for (;;) {
                m = w.face(px, py, next);
                if (w.lin == goal || m >= rem || nseg >= (unsigned)g.max_steps) break;
                ++nseg;
                if (m > 0.f) atomicAdd(gc + w.lin, s * m);
                rem -= m;
                if (left.out(px, py)) {
                    m = -1.f;
                    break;
                }
                w.cross(m, px, py, next);
            }
            if (m >= 0.f) {  // the last voxel
                ++nseg;
                if (w.lin == goal) m = fmaxf(camera_leg(g, cm, w, d, p), 0.f);
                m = fminf(m, rem);
                if (m > 0.f) atomicAdd(gc + w.lin, s * m);
            }
        }
    }
    if (stats) block_count(stats, MST_ST_LOSADJ_SEGMENTS, nseg);
}

// Q_c(k): number of sub-pixel rays through voxel k; a ray counts when its chord is at least
// 1e-4 of the smallest voxel edge (grazing rays with chords ~ 0 are not counted)
__global__ void __launch_bounds__(kTB) k_ray_counts(const Geo g, const CamSet cs, const Halton hs, float* __restrict__ Q,
                                                    int total_pix) {
    const float eps = 1e-4f * fminf(g.hx, fminf(g.hy, g.hz));
    const int gp = blockIdx.x * blockDim.x + threadIdx.x;
    if (gp >= total_pix) return;
    const int c = cam_of_pixel(cs, gp);
    float* qc = Q + (size_t)c * g.nvox;
    for (int rho = 0; rho < hs.n; ++rho) {
        float3 p, d;
        int ix, iy, iz;
        if (!pixel_ray_start(g, cs.c[c], hs, gp, rho, p, d, ix, iy, iz)) continue;
        PadWalk w(g, p, d, lin_index(g, ix, iy, iz), g.nx, g.nx * g.ny);
        FacesLeft left(g, d, ix, iy, iz);
        for (int n = 0; n <= g.max_steps; ++n) {
            bool px, py;
            int next;
            const float m = w.face(px, py, next);
            if (m >= eps) atomicAdd(qc + w.lin, 1.f);
            if (left.out(px, py)) break;
            w.cross(m, px, py, next);
        }
    }
}

// conditioning weight from counts: mode 1 -> 1 / max(1, Q), mode 2 -> Q
__global__ void k_qweights(float* Q, long long n, int mode) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        Q[i] = mode == 1 ? 1.f / fmaxf(1.f, Q[i]) : Q[i];
}

// a_c(k) = T_c(k) b_c(k) in the [nvox][cp] layout gathered at photon events
__global__ void k_adjoint_tiles(const float* __restrict__ T, const float* __restrict__ bacc, float* __restrict__ adj,
                                int nvox, int C, int cp) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nvox; k += gridDim.x * blockDim.x)
        for (int c0 = 0; c0 < cp; c0 += 4) {  // one 16-byte store per four cameras
            float v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = c0 + j;
                v[j] = c < C ? T[(size_t)c * nvox + k] * bacc[(size_t)c * nvox + k] : 0.f;
            }
            *reinterpret_cast<float4*>(adj + (size_t)k * cp + c0) = make_float4(v[0], v[1], v[2], v[3]);
        }
}

// surrogate: grad(m) = sum_c Q_c(m) [ j_c(m) T_c(m) b_c(m) - gT_c(m) ], j = Lsrc / beta_ref
__global__ void k_combine_surrogate(const double* __restrict__ Lsrc, const float* __restrict__ beta_ref,
                                    const float* __restrict__ T, const float* __restrict__ bacc,
                                    const float* __restrict__ gT, const float* __restrict__ Qw,
                                    double* __restrict__ grad, int nvox, int C) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nvox; k += gridDim.x * blockDim.x) {
        const float br = beta_ref[k];
        double acc = 0.0;
        for (int c = 0; c < C; ++c) {
            const size_t i = (size_t)c * nvox + k;
            const double j = br > 0.f ? Lsrc[i] / (double)br : 0.0;
            const double q = Qw ? (double)Qw[i] : 1.0;
            acc += q * (j * (double)T[i] * (double)bacc[i] - (double)gT[i]);
        }
        grad[k] = acc;
    }
}

// full: grad(m) = gL(m) - sum_c gT_c(m). With the tiles of a stored-event replay (gbrk not NULL), gL
// lacks what the score kernel left in the copies of its brick tile and pass 2 in its padded tile:
// both are added here and cleared (one launch instead of three).
__global__ void k_combine_full(const Geo g, const float* __restrict__ gT, const double* __restrict__ gL,
                               float* __restrict__ gbrk, int copies, float* __restrict__ gacc,
                               double* __restrict__ grad, int C) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < g.nvox; k += gridDim.x * blockDim.x) {
        const int ix = k % g.nx, iy = (k / g.nx) % g.ny, iz = k / (g.nx * g.ny);
        const int at = pad_index(g, ix, iy, iz);
        double acc = gL[k];
        if (gbrk) {
            const size_t nb = (size_t)brick_bins(g);
            float* x = gbrk + brick_bin(g, (unsigned)ix, (unsigned)iy, (unsigned)iz);
            for (int t = 0; t < copies; ++t) {
                const float v = x[t * nb];
                if (v != 0.f) {
                    acc += (double)v;
                    x[t * nb] = 0.f;
                }
            }
            const float v = gacc[at];
            if (v != 0.f) {
                acc += (double)v;
                gacc[at] = 0.f;
            }
        }
        if (gT)  // voxel estimator: the LOS term; the classic estimator has none
            for (int c = 0; c < C; ++c) acc -= (double)gT[(size_t)c * g.nvox + k];
        grad[k] = acc;
    }
}

// Loss of the classic images (Eq. Cost): r = M (i - i_meas), E += sum r^2, resid = dE/di = 2 r.
__global__ void k_classic_resid(const double* __restrict__ img, const double* __restrict__ meas,
                                const uint8_t* __restrict__ mask, double* __restrict__ resid, double* loss, int npix) {
    double e = 0.0;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < npix; p += gridDim.x * blockDim.x) {
        const double r = (mask && !mask[p]) ? 0.0 : img[p] - meas[p];
        resid[p] = 2.0 * r;
        e += r * r;
    }
    e = warp_sum(e);
    if ((threadIdx.x & 31u) == 0u && e != 0.0) atomicAdd(loss, e);
}

// Laplacian of a dense field: out(k) = sum over in-grid 6-neighbours n of (x(n) - x(k))
template <typename TIn>
__device__ __forceinline__ double lap_at(const Geo& g, const TIn* x, int k) {
    const int ix = k % g.nx, iy = (k / g.nx) % g.ny, iz = k / (g.nx * g.ny);
    const double xk = (double)x[k];
    double acc = 0.0;
    if (ix > 0) acc += (double)x[k - 1] - xk;
    if (ix < g.nx - 1) acc += (double)x[k + 1] - xk;
    if (iy > 0) acc += (double)x[k - g.nx] - xk;
    if (iy < g.ny - 1) acc += (double)x[k + g.nx] - xk;
    if (iz > 0) acc += (double)x[k - g.nx * g.ny] - xk;
    if (iz < g.nz - 1) acc += (double)x[k + g.nx * g.ny] - xk;
    return acc;
}

// Psi = |W Lap beta|^2 (W diagonal by altitude: wz[iz], or 1 when wz is NULL); lap <- W^T W Lap beta
__global__ void k_lap1(const Geo g, const float* __restrict__ beta, const double* __restrict__ wz,
                       double* __restrict__ lap, double* psi) {
    double s = 0.0;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < g.nvox; k += gridDim.x * blockDim.x) {
        const double w = wz ? wz[k / (g.nx * g.ny)] : 1.0;
        const double v = w * lap_at(g, beta, k);
        lap[k] = w * v;
        s += v * v;
    }
    s = warp_sum(s);
    if ((threadIdx.x & 31u) == 0u && s != 0.0) atomicAdd(psi, s);
}

__global__ void k_lap2(const Geo g, const double* __restrict__ lap, double eta, double* __restrict__ grad) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < g.nvox; k += gridDim.x * blockDim.x)
        grad[k] += eta * 2.0 * lap_at(g, lap, k);
}

__global__ void k_add_scaled(double* dst, const double* src, double eta) {
    if (threadIdx.x == 0 && blockIdx.x == 0) *dst += eta * (*src);
}

inline int nblocks(long long n, int tb = kTB, int cap = 1 << 20) {
    const long long b = (n + tb - 1) / tb;
    return (int)(b < cap ? (b > 0 ? b : 1) : cap);
}

}  // namespace

cudaError_t launch_stage(const mst_grid* g, const float* beta, const float* air, int dtype, cudaStream_t st) {
    if (!g->ext_pad) {  // mst_transmittance_noalloc: FP32, one species
        if (dtype != 0 || air) return cudaErrorInvalidValue;
        k_stage<<<nblocks(g->geo.nvox, kTB, 8192), kTB, 0, st>>>(beta, static_cast<float*>(g->ext), g->geo.nvox);
        return cudaGetLastError();
    }
    float* tot = air ? g->btot : nullptr;
    const int np = nblocks(g->geo.npad, kTB, 4096);
    if (dtype == 0) k_stage_pad<0><<<np, kTB, 0, st>>>(beta, air, g->ext_pad, tot, g->geo);
    else if (dtype == 1) k_stage_pad<1><<<np, kTB, 0, st>>>(beta, air, g->ext_pad, tot, g->geo);
    else k_stage_pad<2><<<np, kTB, 0, st>>>(beta, air, g->ext_pad, tot, g->geo);
    return cudaGetLastError();
}

cudaError_t launch_add_air(const mst_grid* g, const float* beta, const float* air, float* out, cudaStream_t st) {
    k_add_air<<<nblocks(g->geo.nvox, kTB, 4096), kTB, 0, st>>>(beta, air, out, g->geo.nvox);
    return cudaGetLastError();
}

cudaError_t launch_los(const mst_grid* g, int dtype, const double* L, const double* /*jfix*/, const float* beta_ref,
                       const float* beta, float* T_out, float* R_out, cudaStream_t st) {
    const dim3 nb((g->geo.nvox + kTB - 1) / kTB, g->n_cams);
    auto go = [&](auto kern, const void* ext) {
        kern<<<nb, kTB, 0, st>>>(g->geo, g->cams, ext, L, beta_ref, beta, T_out, R_out, g->stats);
    };
    if (!g->ext_pad) {  // mst_transmittance_noalloc: FP32, T only
        if (dtype != 0 || R_out) return cudaErrorInvalidValue;
        go(k_los<0, false>, g->ext);
    } else if (dtype == 0) {
        go(k_los<0, true>, g->ext_pad);
    } else if (dtype == 1) {
        go(k_los<1, true>, g->ext_pad);
    } else {
        go(k_los<2, true>, g->ext_pad);
    }
    return cudaGetLastError();
}

// blocks of the pixel-ray kernels
static int pixel_ray_blocks(const mst_grid* g) {
    const int pixels = pixel_rays_block(g->n_rays) / g->n_rays;
    return (g->total_pix + pixels - 1) / pixels;
}

cudaError_t launch_images(const mst_grid* g, const float* R, double* images, const double* meas, const uint8_t* mask,
                          double* resid, double* loss, cudaStream_t st) {
    const float inv_nv = (float)(1.0 / (g->n_rays * g->voxel_volume));
    k_images<<<pixel_ray_blocks(g), kRayBlock, 0, st>>>(g->geo, g->cams, g->halton, inv_nv, R, images, meas, mask, resid,
                                                        loss, g->total_pix, g->stats);
    return cudaGetLastError();
}

cudaError_t launch_backproject(const mst_grid* g, const double* resid, float* bacc, cudaStream_t st) {
    const float inv_nv = (float)(1.0 / (g->n_rays * g->voxel_volume));
    const dim3 nb((g->total_pix + kTB - 1) / kTB, g->total_pix / g->n_cams < kRaysApart ? g->n_rays : 1);
    k_backproject<<<nb, kTB, 0, st>>>(g->geo, g->cams, g->halton, inv_nv, resid, bacc, g->total_pix, g->stats);
    return cudaGetLastError();
}

cudaError_t launch_los_adjoint(const mst_grid* g, const float* R, const float* bacc, float* gT, cudaStream_t st) {
    const int nb = (g->geo.nvox + kTB - 1) / kTB;
    if (nb > g->sm_count * (2048 / kTB))
        k_los_adjoint<true><<<nb * g->n_cams, kTB, 0, st>>>(g->geo, g->cams, R, bacc, gT, g->stats);
    else
        k_los_adjoint<false><<<nb * g->n_cams, kTB, 0, st>>>(g->geo, g->cams, R, bacc, gT, g->stats);
    return cudaGetLastError();
}

cudaError_t launch_ray_counts(const mst_grid* g, float* Q, int mode, cudaStream_t st) {
    const long long n = (long long)g->n_cams * g->geo.nvox;
    cudaError_t e = cudaMemsetAsync(Q, 0, sizeof(float) * n, st);
    if (e != cudaSuccess) return e;
    k_ray_counts<<<nblocks(g->total_pix), kTB, 0, st>>>(g->geo, g->cams, g->halton, Q, g->total_pix);
    if (mode == 1 || mode == 2) k_qweights<<<nblocks(n, kTB, 4096), kTB, 0, st>>>(Q, n, mode);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_tiles(const mst_grid* g, const float* T, const float* bacc, float* adj, cudaStream_t st) {
    k_adjoint_tiles<<<nblocks(g->geo.nvox, kTB, 4096), kTB, 0, st>>>(T, bacc, adj, g->geo.nvox, g->n_cams, g->cp);
    return cudaGetLastError();
}

cudaError_t launch_combine_surrogate(const mst_grid* g, const double* Lsrc, const double* /*jfix*/,
                                     const float* beta_ref, const float* /*beta*/, const float* T, const float* bacc,
                                     const float* gT, const float* Qw, double* grad, cudaStream_t st) {
    k_combine_surrogate<<<nblocks(g->geo.nvox, kTB, 4096), kTB, 0, st>>>(Lsrc, beta_ref, T, bacc, gT, Qw, grad,
                                                                         g->geo.nvox, g->n_cams);
    return cudaGetLastError();
}

cudaError_t launch_combine_full(const mst_grid* g, const float* gT, const double* gL, bool tiles, double* grad,
                                cudaStream_t st) {
    k_combine_full<<<nblocks(g->geo.nvox, kTB, 4096), kTB, 0, st>>>(g->geo, gT, gL, tiles ? g->gbrk : nullptr,
                                                                    (int)g->score_tiles, g->gacc, grad, g->n_cams);
    return cudaGetLastError();
}

cudaError_t launch_classic_residual(const mst_grid* g, const double* img, const double* meas, const uint8_t* mask,
                                    double* resid, double* loss, cudaStream_t st) {
    k_classic_resid<<<nblocks(g->total_pix, kTB, 4096), kTB, 0, st>>>(img, meas, mask, resid, loss, g->total_pix);
    return cudaGetLastError();
}

// Sun mask M_c of Eq. Cost: 0 where the pixel's centre ray is within `radius` of the direction
// to the sun (cos of the angle above cos(radius), evaluated in FP64), 1 elsewhere.
__global__ void k_sun_mask(const CamSet cs, double3 to_sun, double cos_r, uint8_t* __restrict__ mask, int npix) {
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < npix; p += gridDim.x * blockDim.x) {
        const int c = cam_of_pixel(cs, p);
        const Cam& cm = cs.c[c];
        const int li = p - cm.pix_off, i = li % cm.w, j = li / cm.w;
        const double x = (2.0 * (i + 0.5) / cm.w - 1.0) * (double)cm.tx;
        const double y = (2.0 * (j + 0.5) / cm.h - 1.0) * (double)cm.ty;
        const double dx = cm.fx + x * cm.rx + y * cm.ux, dy = cm.fy + x * cm.ry + y * cm.uy;
        const double dz = cm.fz + x * cm.rz + y * cm.uz;
        const double cosang = (dx * to_sun.x + dy * to_sun.y + dz * to_sun.z) / sqrt(dx * dx + dy * dy + dz * dz);
        mask[p] = cosang > cos_r ? 0 : 1;
    }
}

cudaError_t launch_sun_mask(const mst_grid* g, double zenith, double azimuth, double radius, uint8_t* mask,
                            cudaStream_t st) {
    const double3 s = make_double3(std::sin(zenith) * std::cos(azimuth), std::sin(zenith) * std::sin(azimuth),
                                   std::cos(zenith));
    k_sun_mask<<<nblocks(g->total_pix, kTB, 4096), kTB, 0, st>>>(g->cams, s, std::cos(radius), mask, g->total_pix);
    return cudaGetLastError();
}

// Eq. channelBeta: the aerosol of channel mu, sigma~_mu times the reference field (FP64 product,
// rounded to FP32 like every beta the library reads).
__global__ void k_channel_beta(const float* __restrict__ ref, double sigma, float* __restrict__ out, int nvox) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nvox; k += gridDim.x * blockDim.x)
        out[k] = (float)(sigma * (double)ref[k]);
}

// Eq. divCost1 and Eq. Cost over channels: grad += sigma~_mu dE_mu/dbeta_mu, loss += E_mu.
__global__ void k_channel_add(double* __restrict__ grad, double sigma, const double* __restrict__ gmu, int nvox,
                              double* loss, const double* loss_mu) {
    const int k0 = blockIdx.x * blockDim.x + threadIdx.x;
    for (int k = k0; k < nvox; k += gridDim.x * blockDim.x) grad[k] += sigma * gmu[k];
    if (k0 == 0) *loss += *loss_mu;
}

cudaError_t launch_channel_beta(const mst_grid* g, const float* ref, double sigma, float* out, cudaStream_t st) {
    k_channel_beta<<<nblocks(g->geo.nvox, kTB, 4096), kTB, 0, st>>>(ref, sigma, out, g->geo.nvox);
    return cudaGetLastError();
}

cudaError_t launch_channel_add(const mst_grid* g, double* grad, double sigma, const double* gmu, double* loss,
                               const double* loss_mu, cudaStream_t st) {
    k_channel_add<<<nblocks(g->geo.nvox, kTB, 4096), kTB, 0, st>>>(grad, sigma, gmu, g->geo.nvox, loss, loss_mu);
    return cudaGetLastError();
}

cudaError_t launch_regularizer(const mst_grid* g, const float* beta, double eta, double* lap, double* psi, double* loss,
                               double* grad, cudaStream_t st) {
    const int nb = nblocks(g->geo.nvox, kTB, 4096);
    cudaError_t e = cudaMemsetAsync(psi, 0, sizeof(double), st);
    if (e != cudaSuccess) return e;
    k_lap1<<<nb, kTB, 0, st>>>(g->geo, beta, g->reg_wz, lap, psi);
    if (grad) k_lap2<<<nb, kTB, 0, st>>>(g->geo, lap, eta, grad);
    if (loss) k_add_scaled<<<1, 32, 0, st>>>(loss, psi, eta);
    return cudaGetLastError();
}

}  // namespace mst
