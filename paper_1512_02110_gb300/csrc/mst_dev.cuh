// Device-side building blocks of the sm_103a path: counter-based random numbers, the
// Henyey-Greenstein phase function and sampler, direction rotation, the staged extinction
// fetch and the FP32 voxel walk (Amanatides-Woo), whose positions are voxel index + offset
// inside the voxel.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <math_constants.h>
#include <stdint.h>

namespace mst {

constexpr int kMaxCams = 64;
constexpr int kMaxRays = 64;

struct Geo {
    int nx, ny, nz;     // voxels per axis
    float hx, hy, hz;   // voxel size (m)
    float ex, ey, ez;   // grid extent (m)
    int nvox;
    int max_steps;      // nx + ny + nz + 8: no straight walk crosses more voxels
    // The photon flights walk a copy of the grid padded with kHalo voxels on every side
    // ([nz + 4][ny + 4][nx + 4], halo extinction +inf), so that leaving the grid needs no bounds
    // test in the voxel step: the walk stops on the first halo layer's extinction, and the
    // extinction of the voxel after it, loaded one step ahead, still lies inside the array.
    int p0, p01;        // nx + 4, (nx + 4)(ny + 4): strides of the padded grid
    float inv_p0, inv_p01;
    int npad;           // (nx + 4)(ny + 4)(nz + 4)
};

constexpr int kHalo = 2;  // halo layers of the padded grid

struct Cam {
    float px, py, pz;              // centre of projection, grid-local metres
    int ix, iy, iz;                // voxel holding the centre (may lie outside the grid)
    float lx, ly, lz;              // offset of the centre inside that voxel
    int inside;                    // centre inside the grid
    float rx, ry, rz;              // right
    float ux, uy, uz;              // up
    float fx, fy, fz;              // forward
    float tx, ty;                  // tan(fov_x/2), tan(fov_x/2) * H / W
    int w, h, pix_off;
};

// What the local estimates need of two cameras, side by side: (ix, iy, iz) as floats (exact: the
// centre lies within 1e6 voxels of the grid) and the offset (lx, ly, lz).
struct __align__(16) CamPair {
    float2 jx, jy, jz, lx, ly, lz;
};

struct CamSet {
    CamPair pair[kMaxCams / 2];
    int n;
    Cam c[kMaxCams];
};

struct Halton {
    int n;
    float a[kMaxRays], b[kMaxRays];
};

// ------------------------------------------------------------------------------------------
// Philox-4x32-10 (Salmon et al., SC'11): counter (photon lo, photon hi, event, stream), key = seed.

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k.x += 0x9E3779B9u;
            k.y += 0xBB67AE85u;
        }
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    }
    return c;
}

// (2 (x >> 9) + 1) / 2^24: 24 significant bits, exact in FP32, strictly inside (0, 1).
__device__ __forceinline__ float u01(uint32_t x) { return __uint2float_rn(2u * (x >> 9) + 1u) * 5.9604644775390625e-08f; }

// stream 0: the forward transport and its replays; 1 + p: backward paths of global pixel p
__device__ __forceinline__ float4 draws(uint2 key, uint64_t photon, uint32_t event, uint32_t stream = 0u) {
    const uint4 x = philox4x32_10(make_uint4((uint32_t)photon, (uint32_t)(photon >> 32), event, stream), key);
    return make_float4(u01(x.x), u01(x.y), u01(x.z), u01(x.w));
}

// The raw Philox block of a counter, and its four uniforms: draws() in two steps, for callers
// that also use the low bits u01 leaves unused.
__device__ __forceinline__ uint4 draw_bits(uint2 key, uint64_t photon, uint32_t event) {
    return philox4x32_10(make_uint4((uint32_t)photon, (uint32_t)(photon >> 32), event, 0u), key);
}

__device__ __forceinline__ float4 u01x4(uint4 x) { return make_float4(u01(x.x), u01(x.y), u01(x.z), u01(x.w)); }

// ------------------------------------------------------------------------------------------
// Henyey-Greenstein (Eq. Phg) and its inverse CDF (Eq. thetaHG, squared reading).

struct HG {
    float g, k1, a, b;             // P = k1 * (a - b mu)^(-3/2)
    float omg, opg, omg2, tg;      // 1 - g, 1 + g, 1 - g^2, 2 g
    bool iso;
};

__device__ __forceinline__ float hg_phase(const HG& h, float mu) {
    const float den = h.a - h.b * mu;
    const float r = rsqrtf(den);
    return h.k1 * r * r * r;
}

// Inverse CDF of Eq. Phg (squared reading of Eq. thetaHG): cos = (1 + g^2 - s^2) / (2 g) with
// s = (1 - g^2) / (1 - g + 2 g u). 1 - cos and 1 + cos are evaluated in factored form,
//   1 - cos = (1-g)(1-u)(s + 1 - g) / D,  1 + cos = (1+g) u (s + 1 + g) / D,  D = 1 - g + 2 g u,
// so sin = sqrt((1 - cos)(1 + cos)) keeps full FP32 precision for forward scattering, where
// sqrt(1 - cos^2) would cancel. 1 - u is exact for the 24-bit uniforms.
__device__ __forceinline__ void hg_sample(const HG& h, float u, float& ct, float& st) {
    float omc, opc;
    if (h.iso) {
        omc = 2.f * (1.f - u);
        opc = 2.f * u;
    } else {
        const float D = fmaf(h.tg, u, h.omg);  // spelled out, like the multiply-adds of rotate_dir
        const float s = h.omg2 / D;
        omc = h.omg * (1.f - u) * (s + h.omg) / D;
        opc = h.opg * u * (s + h.opg) / D;
    }
    ct = fminf(1.f, fmaxf(-1.f, 0.5f * (opc - omc)));
    st = sqrtf(fmaxf(omc * opc, 0.f));
}

// Rayleigh phase function of air molecules (Eq. Pray): 3 / (16 pi) (1 + mu^2).
__device__ __forceinline__ float rayleigh_phase(float mu) { return 0.05968310365946075f * fmaf(mu, mu, 1.f); }

// Inverse CDF of Eq. Pray (Eq. thetaREY): the CDF of the cosine is (mu^3 + 3 mu + 4) / 8, and
// Cardano's root of mu^3 + 3 mu + 4 - 8u = 0 is mu = c - 1/c with c = cbrt(q + sqrt(q^2 + 1)),
// q = 4u - 2. q + sqrt(q^2 + 1) lies in [0.23, 4.3] for u in [0, 1], so nothing cancels.
__device__ __forceinline__ void rayleigh_sample(float u, float& ct, float& st) {
    const float q = fmaf(4.f, u, -2.f);
    const float c = cbrtf(q + sqrtf(fmaf(q, q, 1.f)));
    ct = fminf(1.f, fmaxf(-1.f, c - 1.f / c));
    st = sqrtf(fmaxf((1.f - ct) * (1.f + ct), 0.f));
}

// New unit direction at polar angle (cos ct, sin st) and azimuth 2 pi u1 about d. Transverse
// frame: e2 = normalize(axis x d), e1 = e2 x d, axis = z unless |d_z| >= 0.9, then x.
// Every multiply-add is spelled out (fmaf, or __fmul_rn which is never fused): the kernels that
// replay a path must compute each direction bit for bit like the forward did, whatever the
// compiler fuses in the code around them.
__device__ __forceinline__ float3 rotate_dir(float3 d, float ct, float st, float u1) {
    float sp, cp;
    sincospif(2.f * u1, &sp, &cp);
    float3 e2;
    if (fabsf(d.z) < 0.9f) {
        const float n = rsqrtf(fmaf(d.x, d.x, __fmul_rn(d.y, d.y)));
        e2 = make_float3(-d.y * n, d.x * n, 0.f);
    } else {
        const float n = rsqrtf(fmaf(d.y, d.y, __fmul_rn(d.z, d.z)));
        e2 = make_float3(0.f, -d.z * n, d.y * n);
    }
    const float3 e1 = make_float3(fmaf(e2.y, d.z, -__fmul_rn(e2.z, d.y)), fmaf(e2.z, d.x, -__fmul_rn(e2.x, d.z)),
                                  fmaf(e2.x, d.y, -__fmul_rn(e2.y, d.x)));
    const float3 o = make_float3(fmaf(st, fmaf(cp, e1.x, __fmul_rn(sp, e2.x)), __fmul_rn(ct, d.x)),
                                 fmaf(st, fmaf(cp, e1.y, __fmul_rn(sp, e2.y)), __fmul_rn(ct, d.y)),
                                 fmaf(st, fmaf(cp, e1.z, __fmul_rn(sp, e2.z)), __fmul_rn(ct, d.z)));
    const float rn = rsqrtf(fmaf(o.x, o.x, fmaf(o.y, o.y, __fmul_rn(o.z, o.z))));
    return make_float3(o.x * rn, o.y * rn, o.z * rn);
}

// ------------------------------------------------------------------------------------------
// Extinction storage: the grid staged in the compute dtype, x fastest ([nz][ny][nx], the
// linear voxel index). A voxel step changes the index by +-1, +-nx or +-nx ny, one multiply-add;
// the whole 64^3 grid is 1 MB and stays in L2, where 8^3 bricks bought no measurable locality
// but cost the walk a wrap test and two selects per step.

__device__ __forceinline__ int lin_index(const Geo& g, int ix, int iy, int iz) { return ix + g.nx * (iy + g.ny * iz); }

// index of voxel (ix, iy, iz) in the padded grid (each index may lie in the halo, -kHalo .. n + kHalo - 1)
__host__ __device__ __forceinline__ int pad_index(const Geo& g, int ix, int iy, int iz) {
    return (ix + kHalo) + g.p0 * (iy + kHalo) + g.p01 * (iz + kHalo);
}

// (ix, iy, iz) of padded index q, each in [-kHalo, n + kHalo). The quotients come from FP32 reciprocals and
// are corrected by one step: q < 2^31 and the quotients are below 2^12, so the FP32 estimate is
// off by at most one.
__device__ __forceinline__ void unpad(const Geo& g, int q, int& ix, int& iy, int& iz) {
    int a = (int)((float)q * g.inv_p01);
    int r = q - a * g.p01;
    if (r < 0) { --a; r += g.p01; } else if (r >= g.p01) { ++a; r -= g.p01; }
    int b = (int)((float)r * g.inv_p0);
    int c = r - b * g.p0;
    if (c < 0) { --b; c += g.p0; } else if (c >= g.p0) { ++b; c -= g.p0; }
    ix = c - kHalo;
    iy = b - kHalo;
    iz = a - kHalo;
}

// linear voxel index k of a padded index; false for a halo voxel
__device__ __forceinline__ bool interior_lin(const Geo& g, int q, int& k) {
    int ix, iy, iz;
    unpad(g, q, ix, iy, iz);
    k = lin_index(g, ix, iy, iz);
    return (unsigned)ix < (unsigned)g.nx && (unsigned)iy < (unsigned)g.ny && (unsigned)iz < (unsigned)g.nz;
}

// The score kernel's gradient tile keeps 2 x 2 x 2 voxels in one 32-byte sector: a straight flight
// crosses two of them per brick on average, and atomics of one instruction on different words of a
// sector go out as one transaction. Bin of voxel (ix, iy, iz), number of bins, voxel of a bin
// (false: a bin past the grid's odd edge).
__host__ __device__ __forceinline__ int brick_bins(const Geo& g) {
    return ((g.nx + 1) >> 1) * ((g.ny + 1) >> 1) * ((g.nz + 1) >> 1) * 8;
}

__device__ __forceinline__ unsigned brick_bin(const Geo& g, unsigned ix, unsigned iy, unsigned iz) {
    const unsigned b = (ix >> 1) + ((g.nx + 1) >> 1) * ((iy >> 1) + ((g.ny + 1) >> 1) * (iz >> 1));
    return b * 8u + (ix & 1u) + 2u * (iy & 1u) + 4u * (iz & 1u);
}

__device__ __forceinline__ bool brick_voxel(const Geo& g, int i, int& k) {
    const int bx = (g.nx + 1) >> 1, by = (g.ny + 1) >> 1, b = i >> 3;
    const int ix = 2 * (b % bx) + (i & 1), iy = 2 * (b / bx % by) + (i >> 1 & 1), iz = 2 * (b / (bx * by)) + (i >> 2 & 1);
    k = lin_index(g, ix, iy, iz);
    return ix < g.nx && iy < g.ny && iz < g.nz;
}

template <int DT>
struct BetaFetch;
template <>
struct BetaFetch<0> {
    typedef float T;
    static __device__ __forceinline__ float get(const void* p, int a) { return __ldg(static_cast<const float*>(p) + a); }
    static __device__ __forceinline__ T make(float v) { return v; }
};
template <>
struct BetaFetch<1> {
    typedef __half T;
    static __device__ __forceinline__ float get(const void* p, int a) {
        return __half2float(__ldg(static_cast<const __half*>(p) + a));
    }
    static __device__ __forceinline__ T make(float v) { return __float2half_rn(v); }
};
template <>
struct BetaFetch<2> {
    typedef __nv_bfloat16 T;
    static __device__ __forceinline__ float get(const void* p, int a) {
        return __bfloat162float(__ldg(static_cast<const __nv_bfloat16*>(p) + a));
    }
    static __device__ __forceinline__ T make(float v) { return __float2bfloat16_rn(v); }
};

constexpr int kWalkOverflow = 6;  // "exit face" of a walk that was abandoned

// A sum of FP32 terms held as an unevaluated pair hi + lo: each addition's rounding error is
// recovered exactly (Knuth's TwoSum, six additions) and summed beside it, so n terms keep about
// 48 - log2(n) bits of the 53 that an FP64 sum keeps. The terms are products rounded to 24 bits, and
// that rounding is what the results show: their distance from a 64-bit evaluation is the same to four
// digits and more with either sum (T 7.07e-7, images 1.70e-7 and 2.97e-7, at 64^3 and 95 x 77 x 61 voxels; haze T
// 3.44e-8, images 6.37e-8), T is the same FP32 number, and images differ by 1e-15 to 3e-14 of a pixel.
// This chip's FP64 pipe takes 2.6e11 conversions with their additions a second against 3.2e13 FP32
// operations, and the ray kernels add one term per voxel segment: k_los took 0.93 ms for 1.8e8
// segments with FP64 sums, 0.32 ms with this and the walk below.
struct PairSum {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float s = __fadd_rn(hi, x);
        const float t = __fsub_rn(s, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)), __fsub_rn(x, t)));
        hi = s;
    }
    // an infinite or NaN sum has no error term
    __device__ __forceinline__ double value() const { return isfinite(lo) ? (double)hi + (double)lo : (double)hi; }
};

// ------------------------------------------------------------------------------------------
// Voxel walk of camera rays and lines of sight, in voxel-local form. A point is (voxel, offset inside
// the voxel); the walk keeps, per axis, the distance along the ray from the current point to the next
// face (t), the distance between faces (q = h / |d|) and the change of the voxel's index at a crossing. A
// step of length s subtracts s from two axes and resets the crossed one to q, so every quantity
// stays of the size of one voxel and FP32 keeps ~1e-6 m resolution however large the grid. Ties go to x,
// then y, then z. The index runs over the padded grid, whose halo tells the walk that it has left, or
// over the linear one beside a FacesLeft.
struct PadWalk {
    float tx, ty, tz, qx, qy, qz;
    int dx, dy, dz, lin;

    PadWalk() = default;
    static __host__ __device__ __forceinline__ void axis(float p, float d, float h, int stride, float& t, float& q, int& dl) {
        int s;  // (the stride set in the branches instead: 2 % slower lines of sight)
        if (d > 0.f) {
            const float inv = 1.f / d;
            t = (h - p) * inv;
            q = h * inv;
            s = 1;
        } else if (d < 0.f) {
            const float inv = 1.f / -d;
            t = p * inv;
            q = h * inv;
            s = -1;
        } else {
            t = INFINITY;
            q = INFINITY;
            s = 0;
        }
        dl = s * stride;
    }
    // from offset p of voxel `at` of a grid with the strides 1, sy, sz
    __host__ __device__ __forceinline__ PadWalk(const Geo& g, float3 p, float3 d, int at, int sy, int sz) : lin(at) {
        axis(fminf(fmaxf(p.x, 0.f), g.hx), d.x, g.hx, 1, tx, qx, dx);
        axis(fminf(fmaxf(p.y, 0.f), g.hy), d.y, g.hy, sy, ty, qy, dy);
        axis(fminf(fmaxf(p.z, 0.f), g.hz), d.z, g.hz, sz, tz, qz, dz);
    }
    // distance to the next face, the axis it belongs to (ties to x, then y, then z), the voxel behind it
    __host__ __device__ __forceinline__ float face(bool& px, bool& py, int& next) const {
        const float m = fminf(tx, fminf(ty, tz));
        px = tx <= m;
        py = !px && ty <= m;
        next = lin + (px ? dx : (py ? dy : dz));
        return m;
    }
    __host__ __device__ __forceinline__ void cross(float m, bool px, bool py, int next) {
        tx = px ? qx : tx - m;
        ty = py ? qy : ty - m;
        tz = (px || py) ? tz - m : qz;
        lin = next;
    }
};

__host__ __device__ __forceinline__ PadWalk pad_walk(const Geo& g, float3 p, float3 d, int ix, int iy, int iz) {
    return PadWalk(g, p, d, pad_index(g, ix, iy, iz), g.p0, g.p01);
}

// Faces left to the grid's boundary on each axis of a ray that starts in voxel (ix, iy, iz) along d: how
// a walk that reads no field on its way knows that it has left the grid.
struct FacesLeft {
    int x, y, z;
    __device__ __forceinline__ FacesLeft(const Geo& g, float3 d, int ix, int iy, int iz)
        : x(d.x > 0.f ? g.nx - 1 - ix : ix), y(d.y > 0.f ? g.ny - 1 - iy : iy), z(d.z > 0.f ? g.nz - 1 - iz : iz) {}
    // after crossing a face of x (px), of y (py) or of z: whether that was the boundary
    __device__ __forceinline__ bool out(bool px, bool py) {
        x -= px ? 1 : 0;
        y -= py ? 1 : 0;
        z -= px || py ? 0 : 1;
        return (x | y | z) < 0;
    }
};

// Whether a ray on the padded grid ends in a voxel of extinction b and optical depth bs = b * (distance to
// the next face): a flight where its free path tau is not above bs, another ray in the halo (b = +inf). A
// ray that leaves the grid exactly on a voxel's edge crosses its first halo voxel over no distance, where bs
// is inf * 0 = NaN: not above is true there, at most would be false, and the walk would go on past the
// array. (Testing the halo for both kinds costs the backward paths 3 %.)
__host__ __device__ __forceinline__ bool ray_ends(bool flight, float tau, float b, float bs) {
    return flight ? !(tau > bs) : isinf(b);
}

// vector from the point (voxel i, offset p) to the point (voxel j, offset q)
__device__ __forceinline__ float3 local_delta(const Geo& g, int ix, int iy, int iz, float3 p, int jx, int jy, int jz,
                                              float3 q) {
    return make_float3((float)(jx - ix) * g.hx + (q.x - p.x), (float)(jy - iy) * g.hy + (q.y - p.y),
                       (float)(jz - iz) * g.hz + (q.z - p.z));
}

__device__ __forceinline__ int coord_vox(float x, float h, int n) {
    const float f = floorf(x / h);
    return f < 0.f ? 0 : (f > (float)(n - 1) ? n - 1 : (int)f);
}

__device__ __forceinline__ float3 pixel_dir(const Cam& c, float px, float py) {
    const float x = (2.f * px / (float)c.w - 1.f) * c.tx;
    const float y = (2.f * py / (float)c.h - 1.f) * c.ty;
    float3 d = make_float3(c.fx + x * c.rx + y * c.ux, c.fy + x * c.ry + y * c.uy, c.fz + x * c.rz + y * c.uz);
    const float n = 1.f / sqrtf(d.x * d.x + d.y * d.y + d.z * d.z);
    return make_float3(d.x * n, d.y * n, d.z * n);
}

// Start of a ray from a camera: inside the grid it starts at the camera's own voxel and offset;
// outside, the ray is clipped to the grid box (entry point in grid-local metres). Returns
// false if it misses the grid.
__device__ __forceinline__ bool ray_start(const Geo& g, const Cam& c, float3 d, float3& p, int& ix, int& iy, int& iz) {
    if (c.inside) {
        ix = c.ix; iy = c.iy; iz = c.iz;
        p = make_float3(c.lx, c.ly, c.lz);
        return true;
    }
    // Clip to the grid box in a frame at the corner of the camera's voxel (cell index c.i, which
    // may lie outside the grid): the camera is at offset c.l there and the faces the ray enters
    // through are near, so the entry point keeps FP32's resolution however far the grid extends
    // (grid-local coordinates would carry ~1 mm of rounding 10 km from the origin).
    const int ci[3] = {c.ix, c.iy, c.iz}, nn[3] = {g.nx, g.ny, g.nz};
    const float oo[3] = {c.lx, c.ly, c.lz}, dd[3] = {d.x, d.y, d.z}, hh[3] = {g.hx, g.hy, g.hz};
    float tn = 0.f, tf = CUDART_INF_F;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float lo = -(float)ci[a] * hh[a], hi = (float)(nn[a] - ci[a]) * hh[a];
        if (dd[a] == 0.f) {
            if (oo[a] < lo || oo[a] > hi) return false;
        } else {
            float t1 = (lo - oo[a]) / dd[a], t2 = (hi - oo[a]) / dd[a];
            if (t1 > t2) { const float tt = t1; t1 = t2; t2 = tt; }
            tn = fmaxf(tn, t1);
            tf = fminf(tf, t2);
        }
    }
    if (!(tn < tf)) return false;
    int iv[3];
    float pv[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float e = oo[a] + tn * dd[a];  // entry point relative to the camera voxel's corner
        const int k = min(max(ci[a] + (int)floorf(e / hh[a]), 0), nn[a] - 1);
        iv[a] = k;
        pv[a] = e - (float)(k - ci[a]) * hh[a];
    }
    ix = iv[0]; iy = iv[1]; iz = iv[2];
    p = make_float3(pv[0], pv[1], pv[2]);
    return true;
}

__device__ __forceinline__ int cam_of_pixel(const CamSet& cs, int gp) {
    int c = 0;
    for (int i = 1; i < cs.n; ++i)
        if (gp >= cs.c[i].pix_off) c = i;
    return c;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_sumf(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ unsigned long long warp_sumu(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

}  // namespace mst
