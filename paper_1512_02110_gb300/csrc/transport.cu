// Photon transport on the GPU: the forward MC life cycle (Sec. 2.1.2, steps i-vi) with the
// voxelised local estimate of Eq. Lcupdate (k_forward) or the classic one of Eq. fle
// (k_transport), and the score-function gradient of the estimate: from the events the forward
// stored (k_score), or, for the classic estimate and when the events are not held, by two passes
// that walk the photons again from their Philox keys (k_transport).
//
// Work distribution: persistent grids sized to the SM count; warps take photons in batches from a
// global ticket (the score kernel: a forward warp's list of records) until none are left.
#include <algorithm>
#include <type_traits>

#include "mst_internal.h"

namespace mst {
namespace {

constexpr int kTB = 256;
constexpr int kFT = kTransportWarps * 32;  // threads of a forward or score block
constexpr unsigned kFull = 0xffffffffu;
constexpr uint32_t kFnvOffset = 2166136261u;
constexpr uint32_t kFnvPrime = 16777619u;

struct Photon {
    float3 p, d;     // offset inside voxel (ix, iy, iz) and unit direction
    int ix, iy, iz;
    float I, tau;
    uint32_t s;      // scattering events so far
    uint32_t hash;   // forward: path checksum
    uint64_t id;     // global photon id (Philox counter)
    uint32_t idx;    // call-relative index (hash / skip arrays)
};

// Photon tallies of the forward render: per-thread totals, reduced over the warp at the end.
struct Tally {
    float esc[6];
    float absorbed, killed, gained, forced, launched;
    unsigned capped, escaped, traced, lost;
};

// The forward render keeps its tallies in shared memory, one slot per thread (stride kTB
// words, so a warp's lanes touch consecutive words): no atomics and no registers held across
// the voxel loop. The replay passes keep none: their NoTally compiles every update away.
struct LaneTally {
    float* f;  // 11 float fields at f[q * kTB]
    unsigned* u;  // 4 counters at u[q * kTB]
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int q = 0; q < 11; ++q) f[q * kTB] = 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) u[q * kTB] = 0u;
    }
    __device__ __forceinline__ void add_absorbed(float v) { f[6 * kTB] += v; }
    __device__ __forceinline__ void add_killed(float v) { f[7 * kTB] += v; }
    __device__ __forceinline__ void add_gained(float v) { f[8 * kTB] += v; }
    __device__ __forceinline__ void add_forced(float v) { f[9 * kTB] += v; }
    __device__ __forceinline__ void add_capped() { u[0] += 1u; }
    __device__ __forceinline__ void add_launch(float i0) {
        f[10 * kTB] += i0;
        u[2 * kTB] += 1u;
    }
    __device__ __forceinline__ void add_escape(int face, float v) {
        if (face < 6) f[face * kTB] += v;
        if (face == kWalkOverflow) u[3 * kTB] += 1u;
        else u[1 * kTB] += 1u;
    }
    __device__ __forceinline__ Tally load() const {
        Tally t;
#pragma unroll
        for (int q = 0; q < 6; ++q) t.esc[q] = f[q * kTB];
        t.absorbed = f[6 * kTB];
        t.killed = f[7 * kTB];
        t.gained = f[8 * kTB];
        t.forced = f[9 * kTB];
        t.launched = f[10 * kTB];
        t.capped = u[0];
        t.escaped = u[1 * kTB];
        t.traced = u[2 * kTB];
        t.lost = u[3 * kTB];
        return t;
    }
};

// A per-thread event counter that exists only when ON (the one-species kernels carry none).
template <bool ON>
struct EventCount {
    unsigned n = 0u;
    __device__ __forceinline__ void add() { ++n; }
    __device__ __forceinline__ void flush(double* slot, unsigned lane) const {
        const unsigned long long s = warp_sumu(n);
        if (lane == 0u && s) atomicAdd(slot, (double)s);
    }
};
template <>
struct EventCount<false> {
    __device__ __forceinline__ void add() {}
    __device__ __forceinline__ void flush(double*, unsigned) const {}
};

struct NoTally {
    __device__ __forceinline__ void zero() {}
    __device__ __forceinline__ void add_absorbed(float) {}
    __device__ __forceinline__ void add_forced(float) {}
    __device__ __forceinline__ void add_gained(float) {}
    __device__ __forceinline__ void add_killed(float) {}
    __device__ __forceinline__ void add_capped() {}
    __device__ __forceinline__ void add_launch(float) {}
    __device__ __forceinline__ void add_escape(int, float) {}
};

// Voxel and offset of u * n voxels, u = (2m + 1) / 2^24 from a Philox word: (2m + 1) n / 2^24 is
// split exactly in integers, so the offset keeps all 24 bits of u.
__device__ __forceinline__ void launch_coord(uint32_t x, int n, float h, int& i, float& off) {
    const uint64_t q = (uint64_t)(2u * (x >> 9) + 1u) * (uint64_t)n;
    i = (int)(q >> 24);
    off = __uint2float_rn((uint32_t)(q & 0xFFFFFFu)) * 5.9604644775390625e-08f * h;
}

// step i: launch uniformly over the top of the atmosphere along the sun direction, weight I0
__device__ __forceinline__ void launch_photon(const TransportArgs& A, Photon& ph, uint32_t pid) {
    ph.idx = A.out_base + pid;
    ph.id = A.first_id + pid;
    const uint4 x = philox4x32_10(make_uint4((uint32_t)ph.id, (uint32_t)(ph.id >> 32), 0u, 0u), A.key);
    float ox, oy;
    launch_coord(x.x, A.g.nx, A.g.hx, ph.ix, ox);
    launch_coord(x.y, A.g.ny, A.g.hy, ph.iy, oy);
    ph.iz = A.g.nz - 1;
    ph.p = make_float3(ox, oy, A.g.hz);
    ph.d = A.sun;
    ph.I = A.I0;
    ph.tau = -logf(1.f - u01(x.z));  // Eq. taurand
    ph.s = 0u;
    ph.hash = kFnvOffset;
}

// A free flight (steps ii-iii) on the padded grid. Per axis: the distance along the ray from
// the current point to the next face (t), the distance between faces (q = h / |d|), and the change
// of the padded index when a face is crossed (+-1, +-(nx + 4), +-(nx + 4)(ny + 4); 0 for an axis
// the ray does not move along, whose t stays +inf); `lin` is the current voxel's padded index.
// A voxel step subtracts the step from two axes and resets the crossed one to q, so every
// quantity stays of the size of one voxel and FP32 keeps ~1e-6 m resolution anywhere in the grid.
// Ties go to x, then y, then z. Leaving the grid needs no test in the step: the first halo voxel
// has extinction +inf, so its optical depth exceeds any free path and the flight stops there.
// The extinction of the next voxel is loaded one step ahead (bn), so that its latency overlaps
// the current step; the voxel after the first halo layer is the second, still in the array.
struct Flight {
    float tx, ty, tz;
    float qx, qy, qz;
    int dx, dy, dz;
    int lin;
    float bn;  // extinction of voxel lin, loaded ahead
    int left;  // voxel steps left before a flight is abandoned (only a non-finite direction gets there)
};

// 1 / |d| by the hardware reciprocal (__fdividef, within 2 ulp)
__device__ __forceinline__ void flight_axis(float p, float d, float h, int stride, float& t, float& q, int& dl) {
    if (d > 0.f) {
        const float inv = __fdividef(1.f, d);
        t = (h - p) * inv;
        q = h * inv;
        dl = stride;
    } else if (d < 0.f) {
        const float inv = __fdividef(1.f, -d);
        t = p * inv;
        q = h * inv;
        dl = -stride;
    } else {
        t = CUDART_INF_F;
        q = CUDART_INF_F;
        dl = 0;
    }
}

// the flight of photon ph from its point (voxel + offset) along its direction
template <int DT>
__device__ __forceinline__ void flight_init(Flight& f, const TransportArgs& A, const Photon& ph) {
    const Geo& g = A.g;
    flight_axis(fminf(fmaxf(ph.p.x, 0.f), g.hx), ph.d.x, g.hx, 1, f.tx, f.qx, f.dx);
    flight_axis(fminf(fmaxf(ph.p.y, 0.f), g.hy), ph.d.y, g.hy, g.p0, f.ty, f.qy, f.dy);
    flight_axis(fminf(fmaxf(ph.p.z, 0.f), g.hz), ph.d.z, g.hz, g.p01, f.tz, f.qz, f.dz);
    f.lin = pad_index(g, ph.ix, ph.iy, ph.iz);
    f.bn = BetaFetch<DT>::get(A.beta_pad, f.lin);
    f.left = g.max_steps;
}

// One voxel of a free flight (Eq. MCextinct): the free path tau runs out in this voxel when
// tau <= beta * (distance to the next face). Returns true then, or when the voxel is the halo
// (beta = +inf; the caller tells the two apart by b), with b and the face distance m of the voxel;
// false after crossing into the next voxel. SCORE (replay pass 2): every voxel the flight crosses
// receives -S * length in the gradient tile (padded like the grid). The product beta * m is
// rounded on its own (__fmul_rn: never fused into the subtraction that follows), and so is the
// product in flight_offset: the forward and the replay passes are different kernels, and a
// multiply-add fused in one and not in another would send a photon along another path.
template <int DT, bool SCORE>
__device__ __forceinline__ bool flight_step(const TransportArgs& A, Flight& f, float& tau, float& b, float& m, float S,
                                            unsigned& nsc) {
    b = f.bn;
    m = fminf(f.tx, fminf(f.ty, f.tz));
    const bool px = f.tx <= m;
    const bool py = !px && f.ty <= m;
    const int next = f.lin + (px ? f.dx : (py ? f.dy : f.dz));
    f.bn = BetaFetch<DT>::get(A.beta_pad, next);
    const float bs = __fmul_rn(b, m);
    if (!(tau > bs)) return true;
    tau -= bs;
    if (SCORE && S != 0.f && m > 0.f) {
        atomicAdd(A.gacc + f.lin, -S * m);
        ++nsc;
    }
    f.tx = px ? f.qx : f.tx - m;
    f.ty = py ? f.qy : f.ty - m;
    f.tz = (px || py) ? f.tz - m : f.qz;
    f.lin = next;
    return false;
}

// offset along one axis, inside the current voxel, of the point a distance l past the current
// point (d: the direction component; p0: the flight's start offset, kept when d = 0)
__device__ __forceinline__ float flight_offset(float t, float d, float h, float p0, float l) {
    const float v = d > 0.f ? h - __fmul_rn(t - l, d) : (d < 0.f ? (t - l) * -d : p0);
    return fminf(fmaxf(v, 0.f), h);
}

// Exit face (0..5: x-, x+, y-, y+, z-, z+) of a flight that reached halo voxel `lin`.
__device__ __forceinline__ int halo_face(const Geo& g, int lin) {
    int ix, iy, iz;
    unpad(g, lin, ix, iy, iz);
    return ix < 0 ? 0 : (ix >= g.nx ? 1 : (iy < 0 ? 2 : (iy >= g.ny ? 3 : (iz < 0 ? 4 : 5))));
}

// A flight that stopped in voxel f.lin (flight_step returned true) with b, m its extinction and
// face distance: a collision moves the photon to the collision point (offset inside the voxel
// and the voxel's indices) and returns kCollided; the halo returns the exit face. With S != 0 the
// collision voxel receives S * (1/beta - length) (one species) or, with two species (TWO), keeps
// its partial length in ph.tau for the event, which adds S * ([aerosol] / beta_aer - length) once
// the particle is known.
constexpr int kCollided = -2;

template <bool TWO>
__device__ __forceinline__ int flight_end(const TransportArgs& A, Photon& ph, const Flight& f, float tau, float b,
                                          float S, unsigned& nsc) {
    if (isinf(b)) return halo_face(A.g, f.lin);
    const float l = tau / b;
    ph.p = make_float3(flight_offset(f.tx, ph.d.x, A.g.hx, ph.p.x, l), flight_offset(f.ty, ph.d.y, A.g.hy, ph.p.y, l),
                       flight_offset(f.tz, ph.d.z, A.g.hz, ph.p.z, l));
    unpad(A.g, f.lin, ph.ix, ph.iy, ph.iz);
    if (S != 0.f) {
        if constexpr (TWO) {
            ph.tau = l;
        } else {
            atomicAdd(A.gacc + f.lin, S * (1.f / b - l));
            ++nsc;
        }
    }
    return kCollided;
}

// Two FP32 numbers in one 64-bit register: sm_100's packed add, multiply and fused multiply-add take
// one issue slot for both, each rounded as the scalar operation.
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ F2 f2(float2 a) { return f2(a.x, a.y); }
__device__ __forceinline__ void split(F2 a, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v)); }
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
// 1 / sqrt of numbers known to be normal (or of one whose result is not used): no scaling around the unit
__device__ __forceinline__ float rsqrt_normal(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The event side of the local estimates, each value twice: minus the voxel indices (as floats: whole
// numbers below 2^24, so the difference to a camera's is exact) and the offset, the direction, and
// the voxel size.
struct EventPair {
    F2 nx, ny, nz, npx, npy, npz, dx, dy, dz;
    __device__ __forceinline__ EventPair(const Photon& e)
        : nx(f2(-(float)e.ix, -(float)e.ix)), ny(f2(-(float)e.iy, -(float)e.iy)), nz(f2(-(float)e.iz, -(float)e.iz)),
          npx(f2(-e.p.x, -e.p.x)), npy(f2(-e.p.y, -e.p.y)), npz(f2(-e.p.z, -e.p.z)), dx(f2(e.d.x, e.d.x)),
          dy(f2(e.d.y, e.d.y)), dz(f2(e.d.z, e.d.z)) {}
};

// Phase function of the event's particle toward two cameras: Rayleigh (Eq. Pray) for air, HG (Eq.
// Phg) otherwise, of the cosine between the photon's direction and the direction from it to the
// camera. ok: false when the photon sits on the centre of projection (within 1e-19 m: a squared
// distance without a normal FP32 value).
template <bool AIR>
__device__ __forceinline__ F2 phase_pair(const TransportArgs& A, const EventPair& e, const CamPair& c, bool& ok0, bool& ok1) {
    const F2 vx = fma2(f2(c.jx) + e.nx, f2(A.g.hx, A.g.hx), f2(c.lx) + e.npx);
    const F2 vy = fma2(f2(c.jy) + e.ny, f2(A.g.hy, A.g.hy), f2(c.ly) + e.npy);
    const F2 vz = fma2(f2(c.jz) + e.nz, f2(A.g.hz, A.g.hz), f2(c.lz) + e.npz);
    float r0, r1;
    split(fma2(vz, vz, fma2(vx, vx, vy * vy)), r0, r1);
    ok0 = r0 >= 1.17549435e-38f;
    ok1 = r1 >= 1.17549435e-38f;
    const F2 mu = fma2(e.dz, vz, fma2(e.dx, vx, e.dy * vy)) * f2(rsqrt_normal(r0), rsqrt_normal(r1));
    if constexpr (AIR) {
        return f2(0.05968310365946075f, 0.05968310365946075f) * fma2(mu, mu, f2(1.f, 1.f));
    } else {
        // 1 + g^2 - 2 g mu: FP32 numbers near 2 leave no subnormal difference
        split(fma2(f2(-A.hg.b, -A.hg.b), mu, f2(A.hg.a, A.hg.a)), r0, r1);
        const F2 r = f2(rsqrt_normal(r0), rsqrt_normal(r1));
        return f2(A.hg.k1, A.hg.k1) * r * r * r;
    }
}

// Step iv with two species (Sec. 2): the event's particle is air with probability
// beta_air / (beta_air + beta_aer) in its voxel. The uniform comes from the event's own Philox
// block x (the one its scattering draws use): u01 takes the top 23 bits of each word, so the low
// 9 bits of x.x and x.y and the low 5 bits of x.z give a 23-bit m, independent of those draws,
// and u = (2m + 1) / 2^24 (exact in FP32). The test u (beta_air + beta_aer) < beta_air runs in
// FP64 on the FP32 fields, so it takes the same branch as an FP64 evaluation of the same
// expression; an empty aerosol voxel always gives air (u < 1), an empty air voxel aerosol.
__device__ __forceinline__ bool particle_is_air(const TransportArgs& A, uint4 x, int k) {
    const uint32_t m = (x.x & 511u) | ((x.y & 511u) << 9) | ((x.z & 31u) << 18);
    const float u = __uint2float_rn(2u * m + 1u) * 5.9604644775390625e-08f;
    const double ba = (double)__ldg(A.beta_air + k);
    return (double)u * (ba + (double)__ldg(A.beta_aer + k)) < ba;
}

// Eq. Lcupdate: L_c(k) += albedo I_s P(angle between the incoming ray and X_c - X_s), for all
// cameras at once, four cameras per vector atomic into the [nvox][cp] FP32 tile.
template <bool AIR>
__device__ __forceinline__ void le_voxel_p(const TransportArgs& A, const Photon& ph, float w, int k) {
    float* row = A.Lacc + (size_t)k * A.cp;
    const EventPair e(ph);
    const F2 w2 = f2(w, w);
#pragma unroll 1  // (unrolled over 9 cameras, the forward outgrows the instruction cache: 38.1 -> 41.9 ms)
    for (int q = 0; 4 * q < A.cams.n; ++q) {
        float v[4];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            bool ok0, ok1;
            split(w2 * phase_pair<AIR>(A, e, A.cams.pair[2 * q + j], ok0, ok1), v[2 * j], v[2 * j + 1]);
            v[2 * j] = ok0 && 4 * q + 2 * j < A.cams.n ? v[2 * j] : 0.f;
            v[2 * j + 1] = ok1 && 4 * q + 2 * j + 1 < A.cams.n ? v[2 * j + 1] : 0.f;
        }
        atomicAdd(reinterpret_cast<float4*>(row + 4 * q), make_float4(v[0], v[1], v[2], v[3]));
    }
}

__device__ __forceinline__ void le_voxel(const TransportArgs& A, const Photon& ph, float w, int k, bool air) {
    if (air) le_voxel_p<true>(A, ph, w, k);
    else le_voxel_p<false>(A, ph, w, k);
}

// w_s = sum_c a_c(k) albedo I_s P_c(s): the event's contribution to <a, L>.
template <bool AIR>
__device__ __forceinline__ float le_adjoint_p(const TransportArgs& A, const Photon& ph, float w, int k) {
    const float4* row = reinterpret_cast<const float4*>(A.adj + (size_t)k * A.cp);
    const EventPair e(ph);
    const F2 w2 = f2(w, w);
    float acc = 0.f;
    auto two = [&](int pair, float a0, float a1) {  // (the padding's a is 0)
        bool ok0, ok1;
        float v0, v1;
        split(f2(a0, a1) * w2 * phase_pair<AIR>(A, e, A.cams.pair[pair], ok0, ok1), v0, v1);
        acc += ok0 && a0 != 0.f ? v0 : 0.f;
        acc += ok1 && a1 != 0.f ? v1 : 0.f;
    };
    auto group = [&](int q) {
        const float4 a4 = __ldg(row + q);
        two(2 * q, a4.x, a4.y);
        if (4 * q + 2 < A.cams.n) two(2 * q + 1, a4.z, a4.w);
    };
    // the first groups unrolled: their cameras' constants are operands of the arithmetic then
    // instead of loads (score of 3.7e8 events with 9 cameras: 20.8 -> 19.5 ms)
    group(0);
    if (A.cams.n > 4) group(1);
    if (A.cams.n > 8) group(2);
#pragma unroll 1
    for (int q = 3; 4 * q < A.cams.n; ++q) group(q);
    return acc;
}

__device__ __forceinline__ float le_adjoint(const TransportArgs& A, const Photon& ph, float w, int k, bool air) {
    return air ? le_adjoint_p<true>(A, ph, w, k) : le_adjoint_p<false>(A, ph, w, k);
}

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// A shadow ray of Eq. fle: the segment from a point (voxel (ix, iy, iz) + offset p) to camera
// cm's centre, walked on the padded grid like a free flight: per axis the distance to the next
// face (t) and between faces (q), the padded index stride of a crossing, and the length left.
struct Shadow {
    float tx, ty, tz, qx, qy, qz, rem;
    int dx, dy, dz, lin;
};

__device__ __forceinline__ Shadow shadow_init(const Geo& g, int ix, int iy, int iz, float3 p, const Cam& cm) {
    Shadow r;
    const float3 v = local_delta(g, ix, iy, iz, p, cm.ix, cm.iy, cm.iz, make_float3(cm.lx, cm.ly, cm.lz));
    r.rem = sqrtf(v.x * v.x + v.y * v.y + v.z * v.z);
    const float inv = 1.f / r.rem;
    flight_axis(fminf(fmaxf(p.x, 0.f), g.hx), v.x * inv, g.hx, 1, r.tx, r.qx, r.dx);
    flight_axis(fminf(fmaxf(p.y, 0.f), g.hy), v.y * inv, g.hy, g.p0, r.ty, r.qy, r.dy);
    flight_axis(fminf(fmaxf(p.z, 0.f), g.hz), v.z * inv, g.hz, g.p01, r.tz, r.qz, r.dz);
    r.lin = pad_index(g, ix, iy, iz);
    return r;
}

// Its optical depth t_{s->c}. The walk ends at the camera or at the grid's boundary (the first
// halo voxel, extinction +inf: nothing outside the grid attenuates); nvox returns the voxels it
// crossed. The extinction is loaded two voxels ahead: the walk starts, and every step stands, in
// the grid, so the voxel after next lies at most in the second halo layer.
template <int DT>
__device__ __forceinline__ float shadow_tau(const TransportArgs& A, int ix, int iy, int iz, float3 p, const Cam& cm,
                                            unsigned& nvox) {
    Shadow r = shadow_init(A.g, ix, iy, iz, p, cm);
    float tx = r.tx, ty = r.ty, tz = r.tz, rem = r.rem;
    const float qx = r.qx, qy = r.qy, qz = r.qz;
    const int dx = r.dx, dy = r.dy, dz = r.dz;
    int lin = r.lin;
    float bn = BetaFetch<DT>::get(A.beta_pad, lin);
    float bn2;
    {
        const float m = fminf(tx, fminf(ty, tz));
        const bool px = tx <= m;
        const bool py = !px && ty <= m;
        bn2 = BetaFetch<DT>::get(A.beta_pad, lin + (px ? dx : (py ? dy : dz)));
    }
    float tau = 0.f;
#pragma unroll 1
    for (;;) {
        const float b = bn;
        if (isinf(b)) break;
        ++nvox;
        const float m = fminf(tx, fminf(ty, tz));
        const bool px = tx <= m;
        const bool py = !px && ty <= m;
        const int next = lin + (px ? dx : (py ? dy : dz));
        const float ux = px ? qx : tx - m;
        const float uy = py ? qy : ty - m;
        const float uz = (px || py) ? tz - m : qz;
        const float m2 = fminf(ux, fminf(uy, uz));
        const bool px2 = ux <= m2;
        const bool py2 = !px2 && uy <= m2;
        const bool last = !(rem > m);
        float bn3 = 0.f;
        if (!last) bn3 = BetaFetch<DT>::get(A.beta_pad, next + (px2 ? dx : (py2 ? dy : dz)));
        tau += b * (last ? rem : m);
        if (last) break;
        rem -= m;
        tx = ux;
        ty = uy;
        tz = uz;
        lin = next;
        bn = bn2;
        bn2 = bn3;
    }
    return tau;
}

// The shadow-ray terms d f / d beta_m = -f * (length in voxel m): the same walk again, its nvox
// voxels known from shadow_tau, so it loads no extinction; every voxel receives sw * length in
// the gradient tile (padded like the grid).
__device__ __forceinline__ void shadow_scatter(const TransportArgs& A, int ix, int iy, int iz, float3 p, const Cam& cm,
                                               float sw, unsigned nvox) {
    Shadow r = shadow_init(A.g, ix, iy, iz, p, cm);
#pragma unroll 1
    for (unsigned k = 0u; k < nvox; ++k) {
        const float m = fminf(r.tx, fminf(r.ty, r.tz));
        const bool px = r.tx <= m;
        const bool py = !px && r.ty <= m;
        const bool last = !(r.rem > m);
        atomicAdd(A.gacc + r.lin, sw * (last ? r.rem : m));
        if (last) break;
        r.rem -= m;
        r.tx = px ? r.qx : r.tx - m;
        r.ty = py ? r.qy : r.ty - m;
        r.tz = (px || py) ? r.tz - m : r.qz;
        r.lin += px ? r.dx : (py ? r.dy : r.dz);
    }
}

// Where an event lands in camera cm (Eq. fle): false when the camera does not see it (behind
// the camera, outside the image, on the centre, or, with a residual, a pixel of zero residual);
// else the pixel gp and f0 = albedo I_s P(mu) / (|X_c - X_s|^2 Omega_p), times the pixel's
// residual when RES.
template <bool RES>
__device__ __forceinline__ bool classic_pixel(const TransportArgs& A, const Photon& ph, const Cam& cm, float w, bool air,
                                              int& gp, float& f0) {
    const float3 v = local_delta(A.g, cm.ix, cm.iy, cm.iz, make_float3(cm.lx, cm.ly, cm.lz), ph.ix, ph.iy, ph.iz, ph.p);
    const float zc = v.x * cm.fx + v.y * cm.fy + v.z * cm.fz;
    if (!(zc > 0.f)) return false;
    const float x = (v.x * cm.rx + v.y * cm.ry + v.z * cm.rz) / zc;
    const float y = (v.x * cm.ux + v.y * cm.uy + v.z * cm.uz) / zc;
    const float px = floorf((x / cm.tx + 1.f) * 0.5f * (float)cm.w);
    const float py = floorf((y / cm.ty + 1.f) * 0.5f * (float)cm.h);
    if (px < 0.f || py < 0.f || px >= (float)cm.w || py >= (float)cm.h) return false;
    gp = cm.pix_off + (int)py * cm.w + (int)px;
    const float r2 = v.x * v.x + v.y * v.y + v.z * v.z;
    if (!(r2 > 0.f)) return false;
    float cr = 1.f;
    if (RES) {
        cr = (float)A.cres[gp];
        if (cr == 0.f) return false;
    }
    const float mu = -(ph.d.x * v.x + ph.d.y * v.y + ph.d.z * v.z) * rsqrtf(r2);
    f0 = cr * (w * (air ? rayleigh_phase(mu) : hg_phase(A.hg, mu)) / (r2 * A.omega[gp]));
    return true;
}

// Per-warp scratch of the classic estimate, in shared memory: for a group of kClassicGroup
// cameras, each (event lane, camera) pair's value f (res) and pixel (pix), and the list of shadow
// rays to walk (job: event lane | camera in the group << 5); per lane, the voxel segments its
// shadow rays walked, and the warp's count of shadow rays (MST_ST_SHADOW_*).
constexpr int kClassicGroup = 8;
constexpr int kClassicWords = kClassicGroup * 32 * 2 + kClassicGroup * 32 / 4 + 32 + 4;  // per warp
struct ClassicScratch {
    float* res;      // [kClassicGroup][32]
    int* pix;        // [kClassicGroup][32]
    uint8_t* job;    // [kClassicGroup * 32]
    unsigned* seg;   // [32]
    unsigned* rays;  // [1]
};

// Eq. fle for the warp's round of events (lane i < n holds event i; act says whether this lane
// holds one), shadow rays issued warp-coherently: the lanes first find, camera by camera, which
// cameras see their event and compact those (event, camera) pairs into a list; then every lane
// walks one shadow ray of the list at a time, 32 rays per pass over the list, so the warp's lanes
// stay busy however few cameras see each event. OP 0 adds each f = f0 exp(-t) to its pixel of
// the classic image; OP 1 returns w_s = sum_c cres[p] f (the event's share of <dE/di, i>, for the
// classic-estimator gradient), summed over the cameras in their order; OP 2 also scatters the
// shadow-ray terms -cres[p] f * (length in voxel m) into the gradient tile.
template <int DT, int OP>
__device__ __forceinline__ float le_classic(const TransportArgs& A, const Photon& e, float w, bool air, bool act,
                                            const ClassicScratch& cs) {
    const unsigned lane = threadIdx.x & 31u;
    const uint32_t vox = (uint32_t)e.ix | ((uint32_t)e.iy << 11) | ((uint32_t)e.iz << 22);
    float acc = 0.f;
    for (int c0 = 0; c0 < A.cams.n; c0 += kClassicGroup) {
        const int gn = min(kClassicGroup, A.cams.n - c0);
        int qn = 0;
        for (int cl = 0; cl < gn; ++cl) {
            int gp = 0;
            float f0 = 0.f;
            const bool vis = act && classic_pixel<(OP > 0)>(A, e, A.cams.c[c0 + cl], w, air, gp, f0);
            cs.res[cl * 32 + lane] = vis ? f0 : 0.f;
            if (OP == 0) cs.pix[cl * 32 + lane] = gp;
            const unsigned vm = __ballot_sync(kFull, vis);
            if (vis) cs.job[qn + __popc(vm & lanemask_lt())] = (uint8_t)(lane | ((unsigned)cl << 5));
            qn += __popc(vm);
        }
        if (lane == 0u) *cs.rays += (unsigned)qn;
        __syncwarp();
        for (int j0 = 0; j0 < qn; j0 += 32) {
            const int j = j0 + (int)lane;
            const unsigned jb = j < qn ? cs.job[j] : 0u;
            const int el = (int)(jb & 31u), cl = (int)(jb >> 5);
            const uint32_t v = __shfl_sync(kFull, vox, el);
            const float3 p = make_float3(__shfl_sync(kFull, e.p.x, el), __shfl_sync(kFull, e.p.y, el),
                                         __shfl_sync(kFull, e.p.z, el));
            if (j < qn) {
                const Cam& cm = A.cams.c[c0 + cl];
                const int ix = (int)(v & 0x7FFu), iy = (int)((v >> 11) & 0x7FFu), iz = (int)(v >> 22);
                const int r = cl * 32 + el;
                unsigned nv = 0u;
                const float f = cs.res[r] * expf(-shadow_tau<DT>(A, ix, iy, iz, p, cm, nv));
                if (OP == 0) {
                    atomicAdd(A.cimg + cs.pix[r], (double)f);
                } else {
                    cs.res[r] = f;
                    if (OP == 2) shadow_scatter(A, ix, iy, iz, p, cm, -f, nv);
                }
                cs.seg[lane] += OP == 2 ? 2u * nv : nv;
            }
        }
        __syncwarp();
        if (OP > 0)
            for (int cl = 0; cl < gn; ++cl) acc += cs.res[cl * 32 + lane];
        __syncwarp();
    }
    return acc;
}

// step v (albedo weighting, Russian roulette) and step vi (new direction by the particle's
// phase function, next free path). Returns 0 to continue or the termination code.
// PRE: x is the event's Philox block, already drawn (two species: the particle came from it).
template <bool PRE, typename TallyT>
__device__ __forceinline__ int after_event(const TransportArgs& A, Photon& ph, TallyT& t, bool air, uint4 x) {
    const float alb = air ? A.albedo_air : A.albedo;
    t.add_absorbed((1.f - alb) * ph.I);
    ph.I *= alb;
    if (ph.I == 0.f) return 2;
    if (A.max_order > 0 && (int)ph.s >= A.max_order) {
        t.add_forced(ph.I);
        return 4;
    }
    if ((int)ph.s >= A.max_events) {
        t.add_forced(ph.I);
        t.add_capped();
        return 5;
    }
    const float4 u = PRE ? u01x4(x) : draws(A.key, ph.id, ph.s);
    if (ph.I < A.rr_below) {
        if (u.z < A.rr_survival) {
            t.add_gained(ph.I * (A.inv_rr_survival - 1.f));
            ph.I *= A.inv_rr_survival;
        } else {
            t.add_killed(ph.I);
            return 3;
        }
    }
    float ct, st;
    if (air) rayleigh_sample(u.x, ct, st);
    else hg_sample(A.hg, u.x, ct, st);
    ph.d = rotate_dir(ph.d, ct, st, u.y);
    ph.tau = -logf(1.f - u.w);
    return 0;
}

// Debug outputs: a photon's path checksum and the point of its last event (or launch).
__device__ __forceinline__ uint32_t end_hash(uint32_t hash, uint32_t s, int term) {
    return (((hash ^ s) * kFnvPrime) ^ (uint32_t)term) * kFnvPrime;
}

__device__ __forceinline__ void write_point(const TransportArgs& A, const Photon& ph) {
    A.point[ph.idx] = make_float4(ph.p.x, ph.p.y, ph.p.z,
                                  __uint_as_float((uint32_t)ph.ix | ((uint32_t)ph.iy << 11) | ((uint32_t)ph.iz << 22)));
}

__device__ __forceinline__ void finish_photon(const TransportArgs& A, const Photon& ph, int term) {
    if (A.hash) A.hash[ph.idx] = end_hash(ph.hash, ph.s, term);
    if (A.point) write_point(A, ph);
}

// the forward keeps the running checksum in the output itself
__device__ __forceinline__ void finish_hash(const TransportArgs& A, uint32_t idx, uint32_t s, int term) {
    A.hash[idx] = end_hash(A.hash[idx], s, term);
}

// One stored event (forward, full gradient), three 16-byte words: where it happened; the incoming
// direction and albedo * weight; the photon, the event number with the particle (1: air) in bit
// 31, the free path left when the flight entered the event's voxel (e.tau, set at the collision),
// and the record of the photon's previous event (kNoEvent: none), where this event's flight began.
__device__ __forceinline__ void store_event(const TransportArgs& A, unsigned long long i, const Photon& e, float wgt,
                                            bool air, uint32_t prev) {
    uint4* r = A.evrec + i;
    r[0] = make_uint4((uint32_t)e.ix | ((uint32_t)e.iy << 11) | ((uint32_t)e.iz << 22), __float_as_uint(e.p.x),
                      __float_as_uint(e.p.y), __float_as_uint(e.p.z));
    r[A.ev_cap] = make_uint4(__float_as_uint(e.d.x), __float_as_uint(e.d.y), __float_as_uint(e.d.z), __float_as_uint(wgt));
    r[2 * A.ev_cap] = make_uint4(e.idx - A.out_base, e.s | (air ? 0x80000000u : 0u), __float_as_uint(e.tau), prev);
}

// ------------------------------------------------------------------------------------------
// Per-warp photon stacks in shared memory (structure of arrays: lane i touches word i, so
// pushes and pops are free of bank conflicts). A warp holds at most 32 flying photons, fewer
// than 32 queued events once a round of events is done (events are processed 32 at a time as
// soon as 32 are queued) and a ready stack: new photons are launched only when the ready stack
// is empty, so right after a launch a warp holds 32 flying + at most 31 queued photons and never
// more than 63 in total. The event and ready stacks therefore share one array of kSlots = 64
// slots, the events growing up from slot 0 and the ready photons down from slot 63: together
// they never hold more than 63. (Two separate 64-slot stacks took 49 KB of shared memory per
// block of the forward, which the SM's L1 gives up to hold the extinction grid.)

constexpr int kScoreTile = 4096;   // photons per block in the list kernels
// Stored events are written in per-warp chunks of kEvChunk slots (one reservation on the global
// counter per chunk). A warp's photons come from its own ticket batches and all events of a photon
// lie in its warp's chunks in the order they happened, so the score kernel can walk a warp's
// chunks backwards and meet every photon's events from the last to the first. The buffer keeps
// one chunk per resident warp of headroom for the chunks' unused tails.
constexpr unsigned kEvChunk = kEventChunk;
constexpr uint32_t kNoPhoton = 0xFFFFFFFFu;  // photon word of a chunk's unused tail slots
constexpr uint32_t kNoEvent = 0xFFFFFFFFu;   // previous record of a photon's first event
constexpr int kSlots = 64;
// Voxels a flying lane advances per loop trip, and minimum resident blocks per SM (register
// budget), per kernel mode (the forward's and the score's trips: kForwardTrip, kScoreTrip); set from
// sweeps on the 64^3 cumulus workload.
// Classic estimate, forward and replay passes: 6 / 8 / 10 / 12 / 16 voxels a trip ran the forward in
// 8.66 / 8.59 / 9.30 / 9.30 / 8.50 ms (2e6 photons, 9 cameras, 64^3), pass 2 in 24.4 / 25.0 / - / 24.7 / 23.0 at
// 5e5, where the longest photon's chain sets the time, and pass 1 in 3.8 whatever the trip.
constexpr int kStepsClassic = 16;
constexpr int kStepsPass1 = 8;
constexpr int kStepsPass2 = 6;
// The forward launches photons when this many slots are free: 1 / 8 / 16 / 24 / 32 ran 37.0 / 36.9 /
// 37.1 / 39.2 / 42.8 ms at 1e8 photons (64^3): waiting for more leaves lanes idle.
constexpr int kLaunchFrom = 8;
constexpr int kMinBlocksForward = 4;
constexpr int kMinBlocksScore = 4;
constexpr int kMinBlocksClassic = 3;
constexpr int kMinBlocksPass1 = 3;
constexpr int kMinBlocksPass2 = 3;

// kernel modes
// kFwdVoxel: k_forward; kScore: k_score; kFwdClassic, kPass1, kPass2 and kPass1C, kPass2C: the classic
// forward and the replay passes of the voxelised and the classic estimate (k_transport)
constexpr int kFwdVoxel = 0, kFwdClassic = 1, kPass2 = 2, kPass1 = 3, kScore = 4, kPass1C = 5, kPass2C = 6;

template <int NW>
struct Stack {
    uint32_t* w;  // NW arrays of cap words
    int cap;
};

// words of a stack slot: the photon, and a replay's event count and sum
template <int MODE>
struct Rec {
    static constexpr int NW = MODE >= kPass2 ? 15 : 12;
};

template <int NW>
__device__ __forceinline__ void put(const Stack<NW>& q, int slot, const Photon& ph, uint32_t nev, double acc) {
    uint32_t* b = q.w + slot;
    const int c = q.cap;
    b[0 * c] = __float_as_uint(ph.p.x);
    b[1 * c] = __float_as_uint(ph.p.y);
    b[2 * c] = __float_as_uint(ph.p.z);
    b[3 * c] = __float_as_uint(ph.d.x);
    b[4 * c] = __float_as_uint(ph.d.y);
    b[5 * c] = __float_as_uint(ph.d.z);
    b[6 * c] = (uint32_t)ph.ix | ((uint32_t)ph.iy << 11) | ((uint32_t)ph.iz << 22);
    b[7 * c] = __float_as_uint(ph.I);
    b[8 * c] = __float_as_uint(ph.tau);
    b[9 * c] = ph.s;
    b[10 * c] = ph.hash;
    b[11 * c] = ph.idx;
    if (NW > 12) {
        b[12 * c] = nev;
        b[13 * c] = (uint32_t)__double_as_longlong(acc);
        b[14 * c] = (uint32_t)((unsigned long long)__double_as_longlong(acc) >> 32);
    }
}

template <int NW>
__device__ __forceinline__ void get(const Stack<NW>& q, int slot, const TransportArgs& A, Photon& ph, uint32_t& nev,
                                    double& acc) {
    const uint32_t* b = q.w + slot;
    const int c = q.cap;
    ph.p = make_float3(__uint_as_float(b[0]), __uint_as_float(b[c]), __uint_as_float(b[2 * c]));
    ph.d = make_float3(__uint_as_float(b[3 * c]), __uint_as_float(b[4 * c]), __uint_as_float(b[5 * c]));
    const uint32_t v = b[6 * c];
    ph.ix = (int)(v & 0x7FFu);
    ph.iy = (int)((v >> 11) & 0x7FFu);
    ph.iz = (int)(v >> 22);
    ph.I = __uint_as_float(b[7 * c]);
    ph.tau = __uint_as_float(b[8 * c]);
    ph.s = b[9 * c];
    ph.hash = b[10 * c];
    ph.idx = b[11 * c];
    ph.id = A.first_id + (ph.idx - A.out_base);
    if (NW > 12) {
        nev = b[12 * c];
        acc = __longlong_as_double((long long)((unsigned long long)b[13 * c] | ((unsigned long long)b[14 * c] << 32)));
    } else {
        nev = 0u;
        acc = 0.0;
    }
}

// Two species: the event's Philox block waits in the event's own stack slot (popped, so free
// until the next trip pushes events) while the local estimate runs, instead of in registers.
// Volatile, so the compiler reloads it rather than keeping the words live.
template <int NW>
__device__ __forceinline__ void stash_block(const Stack<NW>& q, int slot, uint4 x) {
    volatile uint32_t* b = q.w + slot;
    const int c = q.cap;
    b[0] = x.x;
    b[c] = x.y;
    b[2 * c] = x.z;
    b[3 * c] = x.w;
}

template <int NW>
__device__ __forceinline__ uint4 unstash_block(const Stack<NW>& q, int slot) {
    const volatile uint32_t* b = q.w + slot;
    const int c = q.cap;
    return make_uint4(b[0], b[c], b[2 * c], b[3 * c]);
}

// One slice of the rolling fold (see kFoldSweep): the warp swaps the slice's FP32 bins to zero
// and adds what it took to the FP64 result. Transport lanes keep adding to the same bins with
// 32-bit atomics, so nothing added is lost; each bin's FP32 partial covers at most one sweep.
template <int MODE>
__device__ __forceinline__ void fold_slice(const TransportArgs& A, uint32_t batch, unsigned lane) {
    if constexpr (MODE == kFwdVoxel || MODE == kPass2 || MODE == kPass2C) {
        if (A.fold_bins == 0u) return;
        const uint64_t i0 = (uint64_t)(batch % A.fold_nslices) * A.fold_slice;
        const uint64_t i1 = min(i0 + A.fold_slice, A.fold_bins);
        const uint64_t k0 = MODE == kFwdVoxel ? i0 / (uint32_t)A.cp : 0u;  // the slice's first row
        const uint32_t o0 = (uint32_t)(i0 - k0 * (uint32_t)A.cp);
        for (uint64_t i = i0 + lane; i < i1; i += 32) {
            if (MODE == kFwdVoxel) {  // L tile [nvox][cp] -> L64 [C][nvox]
                const uint32_t o = o0 + (uint32_t)(i - i0), row = o / (uint32_t)A.cp;
                const uint64_t k = k0 + row;
                const int c = (int)(o - row * (uint32_t)A.cp);
                if (c < A.cams.n) {
                    const float v = atomicExch(A.Lacc + i, 0.f);
                    if (v != 0.f) atomicAdd(A.L64 + (size_t)c * A.g.nvox + k, (double)v);
                }
            } else {  // gradient tile [nvox] -> g64 [nvox]
                const float v = atomicExch(A.gacc + i, 0.f);  // padded tile
                int k;
                if (v != 0.f && interior_lin(A.g, (int)i, k)) atomicAdd(A.g64 + k, (double)v);
            }
        }
    }
}

// Warp-uniform refill from the pool of n work items: lanes without a photon take the next
// items of the warp's slice, lane 0 refilling the slice from the launch's global ticket.
// on_launch(j) starts item j and returns whether the lane now has a photon; on_batch(t0) runs
// on the whole warp after each new batch.
template <typename LaunchFn, typename BatchFn>
__device__ __forceinline__ void refill(const TransportArgs& A, uint32_t n, bool& fly, bool& dry, uint32_t& wbase,
                                       uint32_t& wend, unsigned lane, LaunchFn&& on_launch, BatchFn&& on_batch) {
    unsigned need = __ballot_sync(kFull, !fly);
    while (need != 0u && !dry) {
        if (wbase >= wend) {
            unsigned t0 = 0u;
            if (lane == 0u) t0 = atomicAdd(A.ticket, (unsigned)kTicketBatch);
            t0 = __shfl_sync(kFull, t0, 0);
            if (t0 >= n) {
                dry = true;
                break;
            }
            wbase = t0;
            wend = min(t0 + (unsigned)kTicketBatch, n);
            on_batch(t0);
        }
        const unsigned rank = __popc(need & lanemask_lt());
        const unsigned avail = wend - wbase;
        if (!fly && rank < avail) fly = on_launch(wbase + rank);
        wbase += min((unsigned)__popc(need), avail);
        need = __ballot_sync(kFull, !fly);
    }
}

__device__ __forceinline__ void flush_tally(const TransportArgs& A, const Tally& t, unsigned segments,
                                            unsigned events, unsigned lane) {
    double v[11];
#pragma unroll
    for (int q = 0; q < 6; ++q) v[q] = warp_sum((double)t.esc[q]);
    v[6] = warp_sum((double)t.absorbed);
    v[7] = warp_sum((double)t.killed);
    v[8] = warp_sum((double)t.gained);
    v[9] = warp_sum((double)t.forced);
    v[10] = warp_sum((double)t.launched);
    const unsigned long long ev = warp_sumu(events), sg = warp_sumu(segments);
    const unsigned long long cap = warp_sumu(t.capped), esc = warp_sumu(t.escaped), tr = warp_sumu(t.traced);
    const unsigned long long lost = warp_sumu(t.lost);
    if (lane == 0u) {
#pragma unroll
        for (int q = 0; q < 6; ++q)
            if (v[q] != 0.0) atomicAdd(A.stats + MST_ST_ESC_XM + q, v[q]);
        atomicAdd(A.stats + MST_ST_ABSORBED, v[6]);
        atomicAdd(A.stats + MST_ST_RR_KILLED, v[7]);
        atomicAdd(A.stats + MST_ST_RR_GAINED, v[8]);
        atomicAdd(A.stats + MST_ST_FORCED, v[9]);
        atomicAdd(A.stats + MST_ST_LAUNCHED, v[10]);
        atomicAdd(A.stats + MST_ST_EVENTS, (double)ev);
        atomicAdd(A.stats + MST_ST_SEGMENTS, (double)sg);
        atomicAdd(A.stats + MST_ST_CAPPED, (double)cap);
        atomicAdd(A.stats + MST_ST_ESCAPED_N, (double)esc);
        atomicAdd(A.stats + MST_ST_TRACED, (double)tr);
        if (lost) atomicAdd(A.stats + MST_ST_LOST, (double)lost);
    }
}

// ------------------------------------------------------------------------------------------
// The classic forward and the replays: the two passes of the adjoint of a classic call, or of one
// whose events are not held. Every loop
// trip (1) fills empty lanes from the ready stack, then from the id pool, (2) advances every flying
// photon by up to TRIP voxels, pushing collisions onto the event stack, and (3) whenever 32 events
// are queued (or the chunk is draining), processes 32 events at once: w_s, albedo, roulette, new
// direction; photons that go on are pushed onto the ready stack. (The forward took the same form
// once; see k_forward for what it gained.)
//
// Two launches per chunk. Pass 1 (MODE 3) walks every photon and stores
// W = sum_s w_s, w_s = sum_c a_c(k_s) albedo I_s P_c(s), and its event count per photon; the
// photons with W != 0 are then gathered into a list, longest first. Pass 2 (MODE 2) walks the
// listed photons again, with S_j = W - sum_{s<j} w_s (FP64), and
// scatters the score of every flight that ends in an event; it stops at pass 1's last event.
// Both passes run the same flight and event arithmetic, so they see the same path.
// TWO: two-species medium (the launch has an air field); one-species kernels carry none of its
// code. TRIP: voxels a flying lane advances per loop trip (0: the mode's default), a compile-time
// constant.
constexpr int min_blocks(int mode) {
    return mode == kPass2 ? kMinBlocksPass2 : (mode == kPass1 ? kMinBlocksPass1 : kMinBlocksClassic);
}

// One scene's photons, run by every warp of the launch until the scene's pool is dry and the
// warp holds none of its photons (flying, queued for an event or ready).
template <int DT, int MODE, bool TWO, int TRIP>
__device__ __forceinline__ void transport_run(const TransportArgs& A, uint32_t* smem) {
    constexpr bool PASS1 = MODE == kPass1 || MODE == kPass1C;
    constexpr bool PASS2 = MODE == kPass2 || MODE == kPass2C;
    constexpr bool CLASSIC = MODE == kFwdClassic || MODE == kPass1C || MODE == kPass2C;
    constexpr bool REPLAY = PASS1 || PASS2;
    constexpr int kStepsPerTrip = TRIP > 0 ? TRIP : (CLASSIC ? kStepsClassic : (PASS2 ? kStepsPass2 : kStepsPass1));
    constexpr int NW = Rec<MODE>::NW;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned warp = threadIdx.x >> 5;
    const Stack<NW> stk{smem + warp * NW * kSlots, kSlots};  // events at slot i, ready photons at kSlots-1-i
    int ev_n = 0, rd_n = 0;  // warp-uniform stack heights

    // photon tallies: forward render only, one shared-memory slot per thread after the stacks
    typename std::conditional<REPLAY, NoTally, LaneTally>::type t;
    if constexpr (!REPLAY) {
        float* tb = reinterpret_cast<float*>(smem + (kTB / 32) * NW * kSlots);
        t.f = tb + threadIdx.x;
        t.u = reinterpret_cast<unsigned*>(tb + 11 * kTB) + threadIdx.x;
    }
    t.zero();
    ClassicScratch cls{};  // the classic estimate's per-warp scratch, after the stacks and tallies
    if constexpr (CLASSIC) {
        uint32_t* cb = smem + (kTB / 32) * NW * kSlots + (REPLAY ? 0 : kTB * 15) + warp * kClassicWords;
        cls.res = reinterpret_cast<float*>(cb);
        cls.pix = reinterpret_cast<int*>(cb + kClassicGroup * 32);
        cls.job = reinterpret_cast<uint8_t*>(cb + 2 * kClassicGroup * 32);
        cls.seg = cb + 2 * kClassicGroup * 32 + kClassicGroup * 8;
        cls.rays = cls.seg + 32;
        cls.seg[lane] = 0u;
        if (lane == 0u) *cls.rays = 0u;
        __syncwarp();
    }

    Photon ph;
    Flight w;
    float tau = 0.f;
    uint32_t nev = 0u;  // pass 2: events of pass 1
    double acc = 0.0;   // pass 1: W; pass 2: S
    bool fly = false, dry = false;
    uint32_t wbase = 0u, wend = 0u;
    unsigned segments = 0u, scatters = 0u, events = 0u;
    EventCount<TWO && !REPLAY> air_events;  // two species: forward events on air
    const uint32_t pool_n = PASS2 ? *A.plist_n : A.n;  // pass 2 walks the list built from pass 1
    // a call whose forward stored its events: the score kernel did the replay unless they did not fit
    if ((PASS1 || MODE == kPass2) && A.ev_cap && *A.ev_count <= A.ev_cap) return;

    for (;;) {
        // (1) fill: ready photons first, new photons only when the ready stack is empty
        unsigned empty = __ballot_sync(kFull, !fly);
        if (empty != 0u && rd_n > 0) {
            const int rank = __popc(empty & lanemask_lt());
            const int take = min(__popc(empty), rd_n);
            if (!fly && rank < take) {
                get(stk, kSlots - rd_n + rank, A, ph, nev, acc);
                flight_init<DT>(w, A, ph);
                tau = ph.tau;
                fly = true;
            }
            rd_n -= take;
            __syncwarp();
        }
        refill(A, pool_n, fly, dry, wbase, wend, lane, [&](uint32_t j) -> bool {
            uint32_t pid = j;
            nev = 0u;
            acc = 0.0;
            if (PASS2) {  // item j of the pass-1 list
                const ScoreRec r = A.plist[j];
                pid = r.pid;
                nev = r.nev;
                acc = r.W;
            } else if (A.skip && A.skip[A.out_base + j]) {
                if (A.hash) A.hash[A.out_base + j] = 0u;
                if (PASS1) A.wbuf[j] = 0.0;
                if (PASS1) A.nevbuf[j] = 0u;
                return false;
            }
            launch_photon(A, ph, pid);
            flight_init<DT>(w, A, ph);
            tau = ph.tau;
            t.add_launch(A.I0);
            return true;
        }, [&](uint32_t t0) { fold_slice<MODE>(A, t0 / (uint32_t)kTicketBatch, lane); });
        const bool any_fly = __any_sync(kFull, fly);
        if (!any_fly && ev_n == 0 && rd_n == 0 && dry) break;

        // (2) up to kStepsPerTrip voxels for every flying photon
        int r = -1;
        if (fly) {
            const float S = PASS2 ? (float)acc : 0.f;
            int nstep = 0;
            bool stop = false;
            float b = 0.f, m = 0.f;
#pragma unroll 1
            while (nstep < kStepsPerTrip) {
                ++nstep;
                if (flight_step<DT, PASS2>(A, w, tau, b, m, S, scatters)) {
                    stop = true;
                    break;
                }
            }
            if (stop) {
                r = flight_end<TWO>(A, ph, w, tau, b, S, scatters);
                if (r >= 0) --nstep;  // the halo voxel is no segment of the path
            }
            segments += nstep;
            // a flight longer than any straight walk through the grid is abandoned
            w.left -= nstep;
            if (r == -1 && w.left < 0) r = kWalkOverflow;
        }
        const bool collided = fly && r == kCollided;
        const unsigned cmask = __ballot_sync(kFull, collided);
        if (collided) {
            put(stk, ev_n + __popc(cmask & lanemask_lt()), ph, nev, acc);
            fly = false;
        } else if (fly && r >= 0) {
            if (REPLAY) {
                if (PASS1) {
                    A.wbuf[ph.idx - A.out_base] = acc;
                    A.nevbuf[ph.idx - A.out_base] = ph.s;
                }
                fly = false;
            } else {
                t.add_escape(r, ph.I);
                finish_photon(A, ph, 1);
                fly = false;
            }
        }
        ev_n += __popc(cmask);
        __syncwarp();

        // (3) events, 32 at a time (fewer only while draining)
        while (ev_n >= 32 || (ev_n > 0 && dry && rd_n == 0 && !__any_sync(kFull, fly))) {
            const int n = min(32, ev_n);
            Photon e;
            uint32_t enev = 0u;
            double eacc = 0.0;
            int term = -1;  // -1 idle lane, 0 goes on, > 0 ended
            if constexpr (CLASSIC) {
                // the classic estimate runs on the whole warp (its shadow rays are spread over all
                // lanes), between the event's per-lane first half and its second
                const bool act = (int)lane < n;
                const int slot = ev_n - 1 - (int)lane;
                bool air = false;
                float wgt = 0.f;
                if (act) {
                    get(stk, slot, A, e, enev, eacc);
                    e.s += 1u;
                    ++events;
                    const int k = lin_index(A.g, e.ix, e.iy, e.iz);
                    if constexpr (TWO) {
                        const uint4 x = draw_bits(A.key, e.id, e.s);
                        air = particle_is_air(A, x, k);
                        stash_block(stk, slot, x);
                    }
                    if (air) air_events.add();
                    wgt = (air ? A.albedo_air : A.albedo) * e.I;
                    if (!REPLAY) e.hash = (e.hash ^ (uint32_t)k) * kFnvPrime;
                }
                const float we = le_classic<DT, REPLAY ? (PASS2 ? 2 : 1) : 0>(A, e, wgt, air, act, cls);
                if (act) {
                    uint4 xb = make_uint4(0u, 0u, 0u, 0u);
                    if constexpr (TWO) xb = unstash_block(stk, slot);
                    if (!REPLAY) {
                        term = after_event<TWO>(A, e, t, air, xb);
                        if (term) finish_photon(A, e, term);
                    } else if (PASS1) {
                        eacc += (double)we;
                        term = after_event<TWO>(A, e, t, air, xb);
                        if (term) {
                            A.wbuf[e.idx - A.out_base] = eacc;
                            A.nevbuf[e.idx - A.out_base] = e.s;
                        }
                    } else {
                        const float S = (float)eacc;  // the score weight of the flight that ended here
                        if (TWO && S != 0.f) {  // two species: the collision voxel's term (see flight_step)
                            atomicAdd(A.gacc + pad_index(A.g, e.ix, e.iy, e.iz),
                                      S * ((air ? 0.f : 1.f / __ldg(A.beta_aer + lin_index(A.g, e.ix, e.iy, e.iz))) -
                                           e.tau));
                            ++scatters;
                        }
                        eacc -= (double)we;
                        term = e.s == enev ? 1 : after_event<TWO>(A, e, t, air, xb);  // stop at pass 1's last event
                    }
                }
            } else {  // the voxelised estimate's replay, per lane
                if ((int)lane < n) {
                    get(stk, ev_n - 1 - (int)lane, A, e, enev, eacc);
                    e.s += 1u;
                    ++events;
                    const int k = lin_index(A.g, e.ix, e.iy, e.iz);
                    const int slot = ev_n - 1 - (int)lane;
                    uint4 xb = make_uint4(0u, 0u, 0u, 0u);  // two species: the event's Philox block
                    bool air = false;
                    if constexpr (TWO) {
                        const uint4 x = draw_bits(A.key, e.id, e.s);
                        air = particle_is_air(A, x, k);
                        stash_block(stk, slot, x);
                    }
                    if (air) air_events.add();
                    const float wgt = (air ? A.albedo_air : A.albedo) * e.I;
                    {
                        const float we = le_adjoint(A, e, wgt, k, air);
                        if (PASS1) {
                            eacc += (double)we;
                            if constexpr (TWO) xb = unstash_block(stk, slot);
                            term = after_event<TWO>(A, e, t, air, xb);
                            if (term) {
                                A.wbuf[e.idx - A.out_base] = eacc;
                                A.nevbuf[e.idx - A.out_base] = e.s;
                            }
                        } else {
                            const float S = (float)eacc;  // the score weight of the flight that ended here
                            if (TWO && S != 0.f) {  // two species: the collision voxel's term (see flight_step)
                                atomicAdd(A.gacc + pad_index(A.g, e.ix, e.iy, e.iz),
                                          S * ((air ? 0.f : 1.f / __ldg(A.beta_aer + k)) - e.tau));
                                ++scatters;
                            }
                            if constexpr (TWO) xb = unstash_block(stk, slot);
                            term = e.s == enev ? 1 : after_event<TWO>(A, e, t, air, xb);  // stop at pass 1's last event
                            eacc -= (double)we;
                        }
                    }
                }
            }
            ev_n -= n;
            __syncwarp();
            const unsigned gmask = __ballot_sync(kFull, term == 0);
            if (term == 0) put(stk, kSlots - 1 - (rd_n + __popc(gmask & lanemask_lt())), e, enev, eacc);
            rd_n += __popc(gmask);
            __syncwarp();
        }
    }
    if constexpr (CLASSIC) {
        const unsigned long long ss = warp_sumu(cls.seg[lane]);
        if (lane == 0u) {
            atomicAdd(A.stats + MST_ST_SHADOW_RAYS, (double)*cls.rays);
            atomicAdd(A.stats + MST_ST_SHADOW_SEGMENTS, (double)ss);
        }
    }
    if constexpr (REPLAY) {
        const unsigned long long ev = warp_sumu(events), sg = warp_sumu(segments), sc = warp_sumu(scatters);
        if (lane == 0u) {
            atomicAdd(A.stats + MST_ST_REPLAY_EVENTS, (double)ev);
            atomicAdd(A.stats + MST_ST_REPLAY_SEGMENTS, (double)sg);
            atomicAdd(A.stats + MST_ST_REPLAY_SCATTERS, (double)sc);
        }
    } else {
        flush_tally(A, t.load(), segments, events, lane);
        air_events.flush(A.stats + MST_ST_AIR_EVENTS, lane);
    }
}

template <int DT, int MODE, bool TWO, int TRIP = 0>
__global__ void __launch_bounds__(kTB, min_blocks(MODE)) k_transport(const TransportArgs A) {
    extern __shared__ uint32_t smem[];
    transport_run<DT, MODE, TWO, TRIP>(A, smem);
}

// Many scenes in one persistent launch (the batched form): every warp runs the scenes one after
// the other from a table in device memory, each until its photons are done, so the launch ends on
// one tail instead of one per scene and small scenes fill the GPU together with large ones.
template <int DT, int MODE, bool TWO, int TRIP = 0>
__global__ void __launch_bounds__(kTB, min_blocks(MODE))
    k_transport_batch(const TransportArgs* __restrict__ scenes, int n_scenes) {
    extern __shared__ uint32_t smem[];
    for (int s = 0; s < n_scenes; ++s) {
        transport_run<DT, MODE, TWO, TRIP>(scenes[s], smem);
        __syncwarp();
    }
}

// ------------------------------------------------------------------------------------------
// The forward render with the voxelised local estimate. A warp owns kSlots photons, each in a slot of
// shared memory for its whole life; lanes walk flights and hold nothing of a photon but its walk.
// Every loop trip (1) launches new photons into free slots when the ready queue runs short, (2) hands
// ready photons to idle lanes, (3) walks every flight by up to TRIP voxels, queueing flights that
// ended in a collision and putting aside those that left the grid, and (4) takes 32 queued
// collisions at once through their event: collision point, record, local estimates, albedo,
// roulette, new direction and the set-up of the next flight, which makes the photon ready again.
//
// A flight is set up and ended where all 32 lanes have one in hand; a lane that begins one only
// loads its walk and stores five words when it ends. (Both used to happen in the walking lanes, ten
// of 32 at a time: 40 % of the kernel's warp instructions, and with a whole photon held in
// registers across the walk.)

// words of a slot: direction (3), weight, events so far, position in the call, previous record, then
// the flight: t (3), free path, padded index, and q (3)
constexpr int kSlotWords = 15;
static_assert(kSlots == 64, "the queues hold slot numbers in bytes");
constexpr int kSD = 0, kSI = 3, kSs = 4, kSIdx = 5, kSPrev = 6, kST = 7, kSTau = 10, kSLin = 11, kSQ = 12;
constexpr int kEscSlots = 64;  // flights out of the grid a warp puts aside

// shared words per warp: the tallies (FP64), slots, escapes (weight, padded index), and the queues
// of slot numbers
constexpr int kFwdWords = 2 * MST_NSTATS + kSlotWords * kSlots + 2 * kEscSlots + 3 * kSlots / 4;
static_assert(kFwdWords % 2 == 0, "the tallies are FP64");

// One axis of a flight as flight_axis sets it up, without its branches; q carries the direction's
// sign. An axis the flight does not move along keeps its offset in q (t = +inf: q is never used there).
__device__ __forceinline__ void ready_axis(float p0, float d, float h, float& t, float& q) {
    const float p = fminf(fmaxf(p0, 0.f), h);
    const float inv = __fdividef(1.f, fabsf(d));
    const float u = (d > 0.f ? h - p : p) * inv;
    t = d == 0.f ? CUDART_INF_F : u;
    q = d == 0.f ? p0 : copysignf(h * inv, d);
}

// What an event adds to the forward's tallies; rare: one of the last four may be set.
struct EventTally {
    float absorbed = 0.f, killed = 0.f, gained = 0.f, forced = 0.f, capped = 0.f;
    bool rare = false;
    __device__ __forceinline__ void add_absorbed(float v) { absorbed = v; }
    __device__ __forceinline__ void add_killed(float v) { killed = v; rare = true; }
    __device__ __forceinline__ void add_gained(float v) { gained = v; rare = true; }
    __device__ __forceinline__ void add_forced(float v) { forced = v; rare = true; }
    __device__ __forceinline__ void add_capped() { capped = 1.f; rare = true; }
};

template <int DT, bool TWO, int TRIP>
__device__ __forceinline__ void forward_run(const TransportArgs& A, uint32_t* smem) {
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    double* tally = reinterpret_cast<double*>(smem + warp * kFwdWords);    // the warp's share of the statistics
    uint32_t* sl = smem + warp * kFwdWords + 2 * MST_NSTATS;               // word f of slot i at sl[f * kSlots + i]
    uint32_t* esc = sl + kSlotWords * kSlots;
    uint8_t* evq = reinterpret_cast<uint8_t*>(esc + 2 * kEscSlots);  // slots of ended flights
    uint8_t* rdq = evq + kSlots;                                     // of ready photons
    uint8_t* frq = rdq + kSlots;                                     // of no photon
    const uint32_t gwarp = blockIdx.x * kTransportWarps + warp;       // the warp's chunk list
    for (int i = (int)lane; i < MST_NSTATS; i += 32) tally[i] = 0.0;
    // adds the lanes' values to a statistic of the warp (nothing when all are 0)
    auto add_tally = [&](int which, float v) {
        if (__any_sync(kFull, v != 0.f)) {
            v = warp_sumf(v);
            if (lane == 0u) tally[which] += (double)v;
        }
    };
    for (int i = (int)lane; i < kSlots; i += 32) frq[i] = (uint8_t)i;
    __syncwarp();

    int ev_n = 0, rd_n = 0, fr_n = kSlots, esc_n = 0;  // warp-uniform queue lengths
    unsigned long long ch_base = ~0ull;                // forward storing events: the warp's current chunk (none yet) ...
    unsigned ch_fill = kEvChunk;                       // ... and its slots in use
    uint32_t wbase = 0u, wend = 0u;                    // photons of the warp's ticket batch not launched yet
    bool dry = false;
    unsigned segments = 0u, events = 0u, launched = 0u, escaped = 0u;
    EventCount<TWO> air_events;

    // the lane's flight
    float tx = 0.f, ty = 0.f, tz = 0.f, qx = 0.f, qy = 0.f, qz = 0.f, tau = 0.f, bn = 0.f;
    int dx = 0, dy = 0, dz = 0, lin = 0, left = 0;
    int slot = -1;  // its photon's slot; -1: no flight

    // a photon in slot i is ready for the flight from offset p of voxel (ix, iy, iz) along d
    auto make_ready = [&](int i, float3 p, float3 d, int ix, int iy, int iz, float free_path) {
        uint32_t* s = sl + i;
        float3 tt, qq;
        ready_axis(p.x, d.x, A.g.hx, tt.x, qq.x);
        ready_axis(p.y, d.y, A.g.hy, tt.y, qq.y);
        ready_axis(p.z, d.z, A.g.hz, tt.z, qq.z);
        s[(kSD + 0) * kSlots] = __float_as_uint(d.x);
        s[(kSD + 1) * kSlots] = __float_as_uint(d.y);
        s[(kSD + 2) * kSlots] = __float_as_uint(d.z);
        s[(kST + 0) * kSlots] = __float_as_uint(tt.x);
        s[(kST + 1) * kSlots] = __float_as_uint(tt.y);
        s[(kST + 2) * kSlots] = __float_as_uint(tt.z);
        s[kSTau * kSlots] = __float_as_uint(free_path);
        s[kSLin * kSlots] = (uint32_t)pad_index(A.g, ix, iy, iz);
        s[(kSQ + 0) * kSlots] = __float_as_uint(qq.x);
        s[(kSQ + 1) * kSlots] = __float_as_uint(qq.y);
        s[(kSQ + 2) * kSlots] = __float_as_uint(qq.z);
    };
    // tallies of up to 32 flights that left the grid, from the end of their queue
    auto count_escapes = [&](int n) {
        int face = -1;
        float I = 0.f;
        if ((int)lane < n) {
            const int i = esc_n - 1 - (int)lane;
            const int at = (int)esc[kEscSlots + i];
            I = __uint_as_float(esc[i]);
            face = at < 0 ? kWalkOverflow : halo_face(A.g, at);
            if (face < kWalkOverflow) ++escaped;
        }
#pragma unroll
        for (int f = 0; f < 6; ++f) add_tally(MST_ST_ESC_XM + f, face == f ? I : 0.f);
        add_tally(MST_ST_LOST, face == kWalkOverflow ? 1.f : 0.f);
        esc_n -= n;
        __syncwarp();
    };
    uint32_t fly = 0u;  // lanes with a flight

    for (;;) {
        const uint32_t idle = ~fly;
        // (1) launch (a few dozen at a time, so that the launch runs with most lanes)
        while (rd_n < __popc(idle) && !dry && (fr_n >= kLaunchFrom || (rd_n == 0 && fly == 0u && ev_n == 0))) {
            if (wbase >= wend) {
                unsigned t0 = 0u;
                if (lane == 0u) t0 = atomicAdd(A.ticket, (unsigned)kTicketBatch);
                t0 = __shfl_sync(kFull, t0, 0);
                if (t0 >= A.n) {
                    dry = true;
                    break;
                }
                wbase = t0;
                wend = min(t0 + (unsigned)kTicketBatch, A.n);
                fold_slice<kFwdVoxel>(A, t0 / (uint32_t)kTicketBatch, lane);
            }
            const int n = min(min(32, fr_n), (int)(wend - wbase));
            bool in = false;
            int i = 0;
            if ((int)lane < n) {
                const uint32_t j = wbase + lane;
                if (A.skip && A.skip[A.out_base + j]) {
                    if (A.hash) A.hash[A.out_base + j] = 0u;
                } else {
                    in = true;
                    i = frq[fr_n - 1 - (int)lane];
                    Photon ph;
                    launch_photon(A, ph, j);
                    make_ready(i, ph.p, ph.d, ph.ix, ph.iy, ph.iz, ph.tau);
                    uint32_t* s = sl + i;
                    s[kSI * kSlots] = __float_as_uint(ph.I);
                    s[kSs * kSlots] = 0u;
                    s[kSIdx * kSlots] = ph.idx;
                    s[kSPrev * kSlots] = kNoEvent;
                    if (A.hash) A.hash[ph.idx] = kFnvOffset;
                    if (A.point) write_point(A, ph);
                    ++launched;
                }
            }
            wbase += (uint32_t)n;
            // skipped photons give their slots back: the launched ones are packed to the top
            const unsigned im = __ballot_sync(kFull, in);
            const unsigned sm = __ballot_sync(kFull, (int)lane < n && !in);
            const int back = (int)lane < n && !in ? frq[fr_n - 1 - (int)lane] : 0;
            __syncwarp();
            if (in) rdq[rd_n + __popc(im & lanemask_lt())] = (uint8_t)i;
            if ((int)lane < n && !in) frq[fr_n - n + __popc(sm & lanemask_lt())] = (uint8_t)back;
            rd_n += __popc(im);
            fr_n += __popc(sm) - n;
            __syncwarp();
        }
        // (2) ready photons to idle lanes
        if (slot < 0) {
            const int r = rd_n - 1 - __popc(idle & lanemask_lt());
            if (r >= 0) {
                slot = rdq[r];
                const uint32_t* s = sl + slot;
                tx = __uint_as_float(s[(kST + 0) * kSlots]);
                ty = __uint_as_float(s[(kST + 1) * kSlots]);
                tz = __uint_as_float(s[(kST + 2) * kSlots]);
                const uint32_t ux = s[(kSQ + 0) * kSlots], uy = s[(kSQ + 1) * kSlots], uz = s[(kSQ + 2) * kSlots];
                qx = fabsf(__uint_as_float(ux));
                qy = fabsf(__uint_as_float(uy));
                qz = fabsf(__uint_as_float(uz));
                tau = __uint_as_float(s[kSTau * kSlots]);
                lin = (int)s[kSLin * kSlots];
                // the sign says which way (an axis without motion is never crossed)
                dx = (int)ux < 0 ? -1 : 1;
                dy = (int)uy < 0 ? -A.g.p0 : A.g.p0;
                dz = (int)uz < 0 ? -A.g.p01 : A.g.p01;
                bn = BetaFetch<DT>::get(A.beta_pad, lin);
                left = A.g.max_steps;
            }
        }
        const int took = min(rd_n, __popc(idle));
        rd_n -= took;
        fly = __ballot_sync(kFull, slot >= 0);
        if (fly == 0u && ev_n == 0) break;  // (dry: a warp without flights has launched what it could)

        // (3) up to TRIP voxels for every flight (see flight_step)
        bool hit = false, out = false;
        float b = 0.f;
        if (slot >= 0) {
            int n = 0;
#pragma unroll 1
            while (n < TRIP) {
                ++n;
                b = bn;
                const float m = fminf(tx, fminf(ty, tz));
                const bool px = tx <= m;
                const bool py = !px && ty <= m;
                const int next = lin + (px ? dx : (py ? dy : dz));
                bn = BetaFetch<DT>::get(A.beta_pad, next);
                const float bs = __fmul_rn(b, m);
                if (!(tau > bs)) {
                    hit = true;
                    break;
                }
                tau -= bs;
                tx = px ? qx : tx - m;
                ty = py ? qy : ty - m;
                tz = (px || py) ? tz - m : qz;
                lin = next;
            }
            out = hit && isinf(b);
            if (out) {
                hit = false;
                --n;  // the halo voxel is no segment of the path
            }
            segments += n;
            left -= n;
            if (!hit && !out && left < 0) {  // longer than any straight walk through the grid
                out = true;
                lin = -1;
            }
        }
        const unsigned hm = __ballot_sync(kFull, hit), om = __ballot_sync(kFull, out);
        if (hit) {
            uint32_t* s = sl + slot;
            s[(kST + 0) * kSlots] = __float_as_uint(tx);
            s[(kST + 1) * kSlots] = __float_as_uint(ty);
            s[(kST + 2) * kSlots] = __float_as_uint(tz);
            s[kSTau * kSlots] = __float_as_uint(tau);
            s[kSLin * kSlots] = (uint32_t)lin;
            evq[ev_n + __popc(hm & lanemask_lt())] = (uint8_t)slot;
            slot = -1;
        }
        ev_n += __popc(hm);
        fly &= ~(hm | om);
        if (om) {
            if (out) {
                const int r = __popc(om & lanemask_lt());
                esc[esc_n + r] = sl[kSI * kSlots + slot];
                esc[kEscSlots + esc_n + r] = (uint32_t)lin;
                frq[fr_n + r] = (uint8_t)slot;
                if (A.hash) finish_hash(A, sl[kSIdx * kSlots + slot], sl[kSs * kSlots + slot], 1);
                slot = -1;
            }
            esc_n += __popc(om);
            fr_n += __popc(om);
            __syncwarp();
            if (esc_n > kEscSlots - 32) count_escapes(32);
        }
        __syncwarp();

        const int fly_n = __popc(fly);
        // (4) events, 32 at a time; while the warp drains, whatever is queued once no photon is ready and the
        // events are no fewer than the flights still under way
        while (ev_n >= 32 || (ev_n > 0 && dry && rd_n == 0 && fly_n <= ev_n)) {
            const int n = min(32, ev_n);
            unsigned long long ev_slot = 0ull;  // storing events: this lane's record slot
            if (A.ev_cap) {
                // the round's slots continue the warp's chunk and spill into a new one
                unsigned long long nb = 0ull;
                if (ch_fill + (unsigned)n > kEvChunk) {  // a new chunk, linked to the warp's last one
                    if (lane == 0u) {
                        nb = atomicAdd(A.ev_count, (unsigned long long)kEvChunk);
                        // (a chunk past the buffer is not linked: the call then replays instead)
                        if (nb + kEvChunk <= A.ev_cap)
                            A.ch_prev[nb / kEvChunk] = ch_base == ~0ull ? kEndChunk : (uint32_t)(ch_base / kEvChunk);
                    }
                    nb = __shfl_sync(kFull, nb, 0);
                }
                const unsigned f = ch_fill + lane;
                ev_slot = f < kEvChunk ? ch_base + f : nb + (f - kEvChunk);
                if (ch_fill + (unsigned)n > kEvChunk) {
                    ch_base = nb;
                    ch_fill = ch_fill + (unsigned)n - kEvChunk;
                } else {
                    ch_fill += (unsigned)n;
                }
            }
            int term = -1;  // -1 idle lane, 0 goes on, > 0 ended
            int i = 0;
            EventTally t;
            if ((int)lane < n) {
                i = evq[ev_n - 1 - (int)lane];
                const uint32_t* s = sl + i;
                Photon e;
                e.d = make_float3(__uint_as_float(s[(kSD + 0) * kSlots]), __uint_as_float(s[(kSD + 1) * kSlots]),
                                  __uint_as_float(s[(kSD + 2) * kSlots]));
                const int at = (int)s[kSLin * kSlots];
                e.tau = __uint_as_float(s[kSTau * kSlots]);
                // the collision point (see flight_end)
                const float l = e.tau / BetaFetch<DT>::get(A.beta_pad, at);
                e.p = make_float3(flight_offset(__uint_as_float(s[(kST + 0) * kSlots]), e.d.x, A.g.hx,
                                                fabsf(__uint_as_float(s[(kSQ + 0) * kSlots])), l),
                                  flight_offset(__uint_as_float(s[(kST + 1) * kSlots]), e.d.y, A.g.hy,
                                                fabsf(__uint_as_float(s[(kSQ + 1) * kSlots])), l),
                                  flight_offset(__uint_as_float(s[(kST + 2) * kSlots]), e.d.z, A.g.hz,
                                                fabsf(__uint_as_float(s[(kSQ + 2) * kSlots])), l));
                unpad(A.g, at, e.ix, e.iy, e.iz);
                e.I = __uint_as_float(s[kSI * kSlots]);
                e.s = s[kSs * kSlots] + 1u;
                e.idx = s[kSIdx * kSlots];
                e.id = A.first_id + (e.idx - A.out_base);
                ++events;
                const int k = lin_index(A.g, e.ix, e.iy, e.iz);
                bool air = false;
                if constexpr (TWO) {
                    // the event's Philox block: its scattering step needs it again, and it waits in
                    // the flight's words meanwhile (volatile, so that no register holds it)
                    const uint4 x = draw_bits(A.key, e.id, e.s);
                    air = particle_is_air(A, x, k);
                    volatile uint32_t* o = sl + i + kST * kSlots;
                    o[0] = x.x;
                    o[kSlots] = x.y;
                    o[2 * kSlots] = x.z;
                    o[3 * kSlots] = x.w;
                }
                if (air) air_events.add();
                const float wgt = (air ? A.albedo_air : A.albedo) * e.I;
                if (A.hash) A.hash[e.idx] = (A.hash[e.idx] ^ (uint32_t)k) * kFnvPrime;
                if (A.point) write_point(A, e);
                if (A.ev_cap && ev_slot < A.ev_cap) store_event(A, ev_slot, e, wgt, air, s[kSPrev * kSlots]);
                le_voxel(A, e, wgt, k, air);
                uint4 xb = make_uint4(0u, 0u, 0u, 0u);
                if constexpr (TWO) {
                    const volatile uint32_t* o = sl + i + kST * kSlots;
                    xb = make_uint4(o[0], o[kSlots], o[2 * kSlots], o[3 * kSlots]);
                }
                term = after_event<TWO>(A, e, t, air, xb);
                if (term == 0) {
                    make_ready(i, e.p, e.d, e.ix, e.iy, e.iz, e.tau);
                    uint32_t* o = sl + i;
                    o[kSI * kSlots] = __float_as_uint(e.I);
                    o[kSs * kSlots] = e.s;
                    o[kSPrev * kSlots] = (uint32_t)ev_slot;
                } else if (A.hash) {
                    finish_hash(A, e.idx, e.s, term);
                }
            }
            ev_n -= n;
            add_tally(MST_ST_ABSORBED, t.absorbed);
            if (__any_sync(kFull, t.rare)) {
                add_tally(MST_ST_RR_KILLED, t.killed);
                add_tally(MST_ST_RR_GAINED, t.gained);
                add_tally(MST_ST_FORCED, t.forced);
                add_tally(MST_ST_CAPPED, t.capped);
            }
            const unsigned gm = __ballot_sync(kFull, term == 0), fm = __ballot_sync(kFull, term > 0);
            if (term == 0) rdq[rd_n + __popc(gm & lanemask_lt())] = (uint8_t)i;
            if (term > 0) frq[fr_n + __popc(fm & lanemask_lt())] = (uint8_t)i;
            rd_n += __popc(gm);
            fr_n += __popc(fm);
            __syncwarp();
        }
    }
    while (esc_n > 0) count_escapes(min(32, esc_n));
    {
        const unsigned long long ev = warp_sumu(events), sg = warp_sumu(segments), la = warp_sumu(launched),
                                 es = warp_sumu(escaped);
        if (lane == 0u) {
            tally[MST_ST_EVENTS] = (double)ev;
            tally[MST_ST_SEGMENTS] = (double)sg;
            tally[MST_ST_TRACED] = (double)la;
            tally[MST_ST_LAUNCHED] = (double)la * (double)A.I0;
            tally[MST_ST_ESCAPED_N] = (double)es;
        }
        __syncwarp();
        for (int i = (int)lane; i < MST_NSTATS; i += 32)
            if (tally[i] != 0.0) atomicAdd(A.stats + i, tally[i]);
        __syncwarp();
    }
    air_events.flush(A.stats + MST_ST_AIR_EVENTS, lane);
    if (A.ev_cap) {  // the warp's last chunk; its tail holds no event
        if (lane == 0u) A.warp_tail[gwarp] = ch_base == ~0ull ? kEndChunk : (uint32_t)(ch_base / kEvChunk);
        if (ch_base != ~0ull)
            for (unsigned f = ch_fill + lane; f < kEvChunk; f += 32u)
                if (ch_base + f < A.ev_cap) A.evrec[2ull * A.ev_cap + ch_base + f].x = kNoPhoton;
    }
}

constexpr size_t forward_smem() {
    return (size_t)kTransportWarps * kFwdWords * sizeof(uint32_t);
}

template <int DT, bool TWO, int TRIP>
__global__ void __launch_bounds__(kFT, kMinBlocksForward) k_forward(const TransportArgs A) {
    extern __shared__ uint32_t smem[];
    forward_run<DT, TWO, TRIP>(A, smem);
}

// Many scenes in one persistent launch: every warp runs the scenes of the table one after another
template <int TRIP>
__global__ void __launch_bounds__(kFT, kMinBlocksForward)
    k_forward_batch(const TransportArgs* __restrict__ scenes, int n_scenes) {
    extern __shared__ uint32_t smem[];
    for (int s = 0; s < n_scenes; ++s) {
        forward_run<0, false, TRIP>(scenes[s], smem);
        __syncwarp();
    }
}

// ------------------------------------------------------------------------------------------
// The score gradient from the stored events. The flight that ended in event s of a photon scores
// S_s = sum_{s' >= s} w_s' (Eq. DirectJacob on the residual), w_s = sum_c a_c(k) albedo I_s P_c(s):
// every voxel it crossed receives -S_s * length, its last voxel S_s (1/beta - length). Each flight is
// told by two records (where the event before it happened, and its own direction, last voxel and
// free path there), so nothing is walked from the Philox keys, and flights need not follow one
// another: a warp takes one forward warp's chunks from the last to the first, so that it meets
// every photon's events in falling order and S is a running sum per photon (FP64), and its lanes
// walk whatever flights are queued.
//
// A batch is 32 records: w_s, S, the last voxel's term, and the flight's set-up (the number of faces
// it crosses is known: the sum of the index differences of its end voxels), queued in shared
// memory; the next batch's records are on their way meanwhile (cp.async). A trip refills idle lanes
// from the queue and walks K voxels per lane; the (bin, term) entries go through a shared-memory
// strip and out transposed, so that one atomic instruction holds consecutive voxels of a few
// flights. Random FP32 atomics run at 2.0e11 a second on this chip whatever the tile's size, but
// the words of one 32-byte sector go out together, and the tile keeps 2 x 2 x 2 voxels in a sector.
// Additions to one bin queue up, so small grids have the tile several times over (score_tiles), a
// block adding to one of the copies.

constexpr int kFlightWords = 10;  // of a queued flight
constexpr int kScoreSlots = 64;   // flights a warp queues: fewer than 32 left when a batch adds 32
constexpr uint32_t kNoEntry = 0xFFFFFFFFu;

template <int K>
constexpr int score_words() {  // shared words per warp: a batch of records, the queue, the strip
    return 3 * 4 * 32 + kFlightWords * kScoreSlots + 2 * 32 * K;
}

// One axis of a score flight: the distance to the next face and between faces, as flight_axis
// computes them, without its branches (32 flights are set up at once).
__device__ __forceinline__ void score_axis(float p, float d, float h, float& t, float& q) {
    const float inv = __fdividef(1.f, fabsf(d));
    p = fminf(fmaxf(p, 0.f), h);
    const float u = (d > 0.f ? h - p : p) * inv;
    t = d == 0.f ? CUDART_INF_F : u;
    q = h * inv;
}

__device__ __forceinline__ void copy16_async(uint32_t* dst, const uint4* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

template <int DT, bool TWO, int K>
__device__ __forceinline__ void score_run(const TransportArgs& A, uint32_t* smem) {
    if (*A.ev_count > A.ev_cap) return;  // the events did not fit: the replay passes run instead
    const unsigned lane = threadIdx.x & 31u;
    uint32_t* rec = smem + (threadIdx.x >> 5) * score_words<K>();  // the lane's record words f at rec[(f * 32 + lane) * 4]
    uint32_t* q = rec + 3 * 4 * 32;                                // queue: word f of slot i at q[f * kScoreSlots + i]
    float2* strip = reinterpret_cast<float2*>(q + kFlightWords * kScoreSlots);
    const unsigned nbins = (unsigned)brick_bins(A.g);
    float* tile = A.gbrk + (size_t)(blockIdx.x % A.score_tiles) * nbins;  // the block's copy
    const uint32_t by8 = 8u * (unsigned)((A.g.nx + 1) >> 1), bz8 = by8 * (unsigned)((A.g.ny + 1) >> 1);
    unsigned stored = 0u, flights = 0u, entries = 0u, lost = 0u;

    // The flight in hand: t and q as in Flight, and per axis the step of its bin (the stride of the
    // bricks, signed, with the axis' bit of the voxel inside the brick). `at` is the bin with the
    // bits of the axes the flight descends mirrored (`flip`): a crossing toggles the axis' bit and
    // enters the next brick when it was set.
    float tx = 0.f, ty = 0.f, tz = 0.f, qx = 0.f, qy = 0.f, qz = 0.f, nS = 0.f;
    uint32_t sx = 0u, sy = 0u, sz = 0u, at = 0u, flip = 0u, goal = 0u;
    int left = 0;  // faces still to cross; 0: no flight

    // the next batch: its records are being copied (pending), or the lists are used up
    uint32_t ch = kEndChunk, prev = kEndChunk;
    int base = -1;
    bool pending = false;
    auto fetch = [&]() {
        if (base < 0) {  // the next chunk of the list, or the next list
            ch = prev;
            while (ch == kEndChunk) {
                unsigned l = 0u;
                if (lane == 0u) l = atomicAdd(A.ticket, 1u);
                l = __shfl_sync(kFull, l, 0);
                if (l >= A.n_warps) break;
                ch = A.warp_tail[l];
            }
            pending = ch != kEndChunk;
            if (!pending) return;
            prev = A.ch_prev[ch];
            base = (int)kEvChunk - 32;
            // one slice of the rolling fold (see kFoldSweep) per chunk
            const uint32_t i0 = ch % A.fold_nslices * A.fold_slice;
            const uint32_t i1 = min(i0 + A.fold_slice, (uint32_t)A.fold_bins);
            for (uint32_t i = i0 + lane; i < i1; i += 32) {
                const float v = atomicExch(A.gbrk + i, 0.f);
                int k;
                if (v != 0.f && brick_voxel(A.g, (int)(i % nbins), k)) atomicAdd(A.g64 + k, (double)v);
            }
        }
        const uint4* r = A.evrec + ((unsigned long long)ch * kEvChunk + (unsigned)base + lane);
#pragma unroll
        for (int f = 0; f < 3; ++f) copy16_async(rec + (f * 32 + lane) * 4, r + f * A.ev_cap);
        asm volatile("cp.async.commit_group;" ::: "memory");
        base -= 32;
        pending = true;
    };
    fetch();

    int qn = 0;  // queued flights (warp-uniform)
    for (;;) {
        const unsigned idle = __ballot_sync(kFull, left == 0);
        const int want = __popc(idle);
        while (qn < want && pending) {  // batches until the queue can fill the idle lanes
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            const uint4 r0 = *reinterpret_cast<const uint4*>(rec + lane * 4);
            const uint4 r1 = *reinterpret_cast<const uint4*>(rec + (32 + lane) * 4);
            const uint4 r2 = *reinterpret_cast<const uint4*>(rec + (64 + lane) * 4);
            const bool on = r2.x != kNoPhoton;
            Photon e;
            e.ix = (int)(r0.x & 2047u);
            e.iy = (int)((r0.x >> 11) & 2047u);
            e.iz = (int)(r0.x >> 22);
            e.p = make_float3(__uint_as_float(r0.y), __uint_as_float(r0.z), __uint_as_float(r0.w));
            e.d = make_float3(__uint_as_float(r1.x), __uint_as_float(r1.y), __uint_as_float(r1.z));
            const bool air = TWO && (r2.y >> 31) != 0u;
            const int k = lin_index(A.g, e.ix, e.iy, e.iz);
            // where the flight began: the previous event, or the launch point
            uint4 o = make_uint4(0u, 0u, 0u, 0u);
            float b = 1.f;
            if (on) {
                if (r2.w != kNoEvent) o = A.evrec[r2.w];
                b = BetaFetch<DT>::get(A.beta_pad, pad_index(A.g, e.ix, e.iy, e.iz));
            }
            fetch();
            const float w = on ? le_adjoint(A, e, __uint_as_float(r1.w), k, air) : 0.f;
            // S: later events first. A batch may hold two events of a photon (rounds of fewer than
            // 32 while the forward's warp drained): they take turns, the later record first.
            const unsigned same = __match_any_sync(kFull, r2.x);
            const int turn = on ? __popc(same & ~(lanemask_lt() | (1u << lane))) : -1;
            const int turns = __reduce_max_sync(kFull, turn);
            double S = 0.0;
            for (int t = 0; t <= turns; ++t) {
                if (turn == t) {
                    S = A.wbuf[r2.x];
                    if (w != 0.f) A.wbuf[r2.x] = S += (double)w;
                }
                __syncwarp();
            }
            const float Sf = (float)S;
            const bool go = on && Sf != 0.f;
            int n = 0;
            if (on && r2.w == kNoEvent) {
                Photon l;
                launch_photon(A, l, r2.x);
                o = make_uint4((uint32_t)l.ix | ((uint32_t)l.iy << 11) | ((uint32_t)l.iz << 22), __float_as_uint(l.p.x),
                               __float_as_uint(l.p.y), __float_as_uint(l.p.z));
            }
            const int ox = (int)(o.x & 2047u), oy = (int)((o.x >> 11) & 2047u), oz = (int)(o.x >> 22);
            const uint32_t bin = brick_bin(A.g, (unsigned)e.ix, (unsigned)e.iy, (unsigned)e.iz);
            if (go) {
                n = abs(e.ix - ox) + abs(e.iy - oy) + abs(e.iz - oz);
                // the last voxel: the length there is the stored free path over the extinction
                const float ib = 1.f / b;
                float is = ib;  // [aerosol] / beta_aer with two species
                if constexpr (TWO) is = air ? 0.f : 1.f / __ldg(A.beta_aer + k);
                atomicAdd(tile + bin, Sf * (is - __uint_as_float(r2.z) * ib));
                ++flights;
                entries += (unsigned)n + 1u;
            }
            if (on) ++stored;
            const unsigned gm = __ballot_sync(kFull, n > 0);
            if (n > 0) {
                float3 t, f;
                score_axis(__uint_as_float(o.y), e.d.x, A.g.hx, t.x, f.x);
                score_axis(__uint_as_float(o.z), e.d.y, A.g.hy, t.y, f.y);
                score_axis(__uint_as_float(o.w), e.d.z, A.g.hz, t.z, f.z);
                const uint32_t fl = (e.d.x < 0.f ? 1u : 0u) | (e.d.y < 0.f ? 2u : 0u) | (e.d.z < 0.f ? 4u : 0u);
                uint32_t* s = q + (qn + __popc(gm & lanemask_lt()));
                s[0] = __float_as_uint(t.x);
                s[1 * kScoreSlots] = __float_as_uint(t.y);
                s[2 * kScoreSlots] = __float_as_uint(t.z);
                s[3 * kScoreSlots] = __float_as_uint(f.x);
                s[4 * kScoreSlots] = __float_as_uint(f.y);
                s[5 * kScoreSlots] = __float_as_uint(f.z);
                s[6 * kScoreSlots] = __float_as_uint(-Sf);
                s[7 * kScoreSlots] = brick_bin(A.g, (unsigned)ox, (unsigned)oy, (unsigned)oz) ^ fl;
                s[8 * kScoreSlots] = bin ^ fl;
                s[9 * kScoreSlots] = (uint32_t)n | (fl << 16);
            }
            qn += __popc(gm);
            __syncwarp();
        }
        if (qn == 0 && want == 32) break;
        // refill from the top of the queue
        if (left == 0) {
            if (at != goal) ++lost;  // a walk that missed its event's voxel (none in valid use)
            goal = at;
            const int slot = qn - 1 - __popc(idle & lanemask_lt());
            if (slot >= 0) {
                const uint32_t* s = q + slot;
                tx = __uint_as_float(s[0]);
                ty = __uint_as_float(s[1 * kScoreSlots]);
                tz = __uint_as_float(s[2 * kScoreSlots]);
                qx = __uint_as_float(s[3 * kScoreSlots]);
                qy = __uint_as_float(s[4 * kScoreSlots]);
                qz = __uint_as_float(s[5 * kScoreSlots]);
                nS = __uint_as_float(s[6 * kScoreSlots]);
                at = s[7 * kScoreSlots];
                goal = s[8 * kScoreSlots];
                const uint32_t nf = s[9 * kScoreSlots];
                left = (int)(nf & 0xFFFFu);
                flip = nf >> 16;
                sx = (flip & 1u ? 0u - 8u : 8u) | 1u;
                sy = (flip & 2u ? 0u - by8 : by8) | 2u;
                sz = (flip & 4u ? 0u - bz8 : bz8) | 4u;
            }
        }
        qn = max(0, qn - want);
        // K voxels per lane into the strip (entry j of a lane at [j][lane ^ 2j]: neither the writes
        // nor the transposed reads meet in a bank)
#pragma unroll
        for (int j = 0; j < K; ++j) {
            uint32_t key = kNoEntry;
            const float m = fminf(tx, fminf(ty, tz));
            if (left > 0) {
                key = at ^ flip;
                const bool px = tx <= m;
                const bool py = !px && ty <= m;
                const uint32_t s = px ? sx : (py ? sy : sz);
                const bool over = (at & s & 7u) != 0u;
                at ^= s & 7u;
                if (over) at += s & ~7u;
                tx = px ? qx : tx - m;
                ty = py ? qy : ty - m;
                tz = (px || py) ? tz - m : qz;
                --left;
            }
            strip[j * 32 + ((lane ^ (2 * j)) & 31)] = make_float2(__uint_as_float(key), nS * m);
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const int i = r * 32 + (int)lane, j = i % K, l = i / K;  // entry j of lane l
            const float2 en = strip[j * 32 + ((l ^ (2 * j)) & 31)];
            const uint32_t key = __float_as_uint(en.x);
            if (key < nbins) atomicAdd(tile + key, en.y);
        }
        __syncwarp();
    }
    const unsigned long long se = warp_sumu(stored), sf = warp_sumu(flights), sn = warp_sumu(entries), sl = warp_sumu(lost);
    if (lane == 0u) {
        if (se) atomicAdd(A.stats + MST_ST_EVENTS_STORED, (double)se);
        atomicAdd(A.stats + MST_ST_REPLAY_EVENTS, (double)sf);
        atomicAdd(A.stats + MST_ST_REPLAY_SEGMENTS, (double)sn);
        atomicAdd(A.stats + MST_ST_REPLAY_SCATTERS, (double)sn);
        if (sl) atomicAdd(A.stats + MST_ST_LOST, (double)sl);
    }
}

template <int DT, bool TWO, int K>
__global__ void __launch_bounds__(kFT, kMinBlocksScore) k_score(const TransportArgs A) {
    extern __shared__ uint32_t smem[];
    score_run<DT, TWO, K>(A, smem);
}

// the batched form: the scenes of a table one after the other
template <int K>
__global__ void __launch_bounds__(kFT, kMinBlocksScore)
    k_score_batch(const TransportArgs* __restrict__ scenes, int n_scenes) {
    extern __shared__ uint32_t smem[];
    for (int s = 0; s < n_scenes; ++s) {
        score_run<0, false, K>(scenes[s], smem);
        __syncwarp();
    }
}

// Pass-2 work list. Photons with W != 0 are binned by their pass-1 event count (the last bin
// takes every count >= kScoreBins - 1) and listed from the highest bin down, so the longest
// replays start first and the launch does not end on a tail of long photons.
__device__ __forceinline__ int score_bin(uint32_t nev) { return (int)min(nev, (uint32_t)(kScoreBins - 1)); }

// Step 1: bin counts cnt[b] over the chunk.
__global__ void __launch_bounds__(kTB) k_score_hist(const double* __restrict__ W, const uint32_t* __restrict__ nev,
                                                    uint32_t n, unsigned* __restrict__ cnt,
                                                    const unsigned long long* ev_count, unsigned long long ev_cap) {
    __shared__ unsigned h[kScoreBins];
    if (ev_cap && *ev_count <= ev_cap) return;  // the score kernel did the replay
    for (int b = threadIdx.x; b < kScoreBins; b += kTB) h[b] = 0u;
    __syncthreads();
    const uint32_t lo = blockIdx.x * kScoreTile, hi = min(lo + (uint32_t)kScoreTile, n);
    for (uint32_t i = lo + threadIdx.x; i < hi; i += kTB) {
        const uint32_t e = nev[i];
        if (e != 0u && W[i] != 0.0) atomicAdd(&h[score_bin(e)], 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kScoreBins; b += kTB)
        if (h[b]) atomicAdd(&cnt[b], h[b]);
}

// Step 2: each tile reserves its slots in every bin (fill[b]) and writes its records there;
// the list length goes to *total.
__global__ void __launch_bounds__(kTB) k_score_scatter(const double* __restrict__ W, const uint32_t* __restrict__ nev,
                                                       uint32_t n, const unsigned* __restrict__ cnt,
                                                       unsigned* __restrict__ fill, unsigned* __restrict__ total,
                                                       ScoreRec* __restrict__ list, const unsigned long long* ev_count,
                                                       unsigned long long ev_cap) {
    __shared__ unsigned h[kScoreBins], pos[kScoreBins];
    if (ev_cap && *ev_count <= ev_cap) return;
    for (int b = threadIdx.x; b < kScoreBins; b += kTB) h[b] = 0u;
    __syncthreads();
    const uint32_t lo = blockIdx.x * kScoreTile, hi = min(lo + (uint32_t)kScoreTile, n);
    for (uint32_t i = lo + threadIdx.x; i < hi; i += kTB) {
        const uint32_t e = nev[i];
        if (e != 0u && W[i] != 0.0) atomicAdd(&h[score_bin(e)], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 32) {  // bin starts, highest bin first: start[b] = sum_{b' > b} cnt[b']
        unsigned run = 0u;
        for (int b0 = kScoreBins - 32; b0 >= 0; b0 -= 32) {
            const int b = b0 + (int)threadIdx.x;
            const unsigned c = cnt[b];
            unsigned incl = c;  // suffix sum within the 32 bins b0 .. b0+31
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned v = __shfl_down_sync(kFull, incl, o);
                if ((int)threadIdx.x + o < 32) incl += v;
            }
            const unsigned start = run + incl - c;
            pos[b] = h[b] ? start + atomicAdd(&fill[b], h[b]) : 0u;
            run += __shfl_sync(kFull, incl, 0);
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) *total = run;
    }
    __syncthreads();
    for (uint32_t i = lo + threadIdx.x; i < hi; i += kTB) {
        const uint32_t e = nev[i];
        const double w = W[i];
        if (e != 0u && w != 0.0) {
            ScoreRec r;
            r.pid = i;
            r.nev = e;
            r.W = w;
            list[atomicAdd(&pos[score_bin(e)], 1u)] = r;
        }
    }
}

// Folds the FP32 L tile [nvox][cp] into the FP64 result [C][nvox] and clears it. A block takes kFoldRows
// rows through shared memory, so that both sides move whole lines (a thread per row read 32 lines
// an instruction: 1.1 ms for 80 x 80 x 120 voxels and 36 cameras).
constexpr int kFoldRows = 32;
__global__ void __launch_bounds__(kTB) k_fold_L(float* __restrict__ Lacc, double* __restrict__ L64, int nvox, int C,
                                                int cp) {
    extern __shared__ float rows[];  // [kFoldRows][cp + 1]
    for (int k0 = blockIdx.x * kFoldRows; k0 < nvox; k0 += gridDim.x * kFoldRows) {
        const int n = min(kFoldRows, nvox - k0);
        float4* from = reinterpret_cast<float4*>(Lacc + (size_t)k0 * cp);
        for (int i = threadIdx.x; i < n * cp / 4; i += kTB) {
            const float4 v = from[i];
            const int row = 4 * i / cp;
            float* to = rows + row * (cp + 1) + (4 * i - row * cp);
            to[0] = v.x;
            to[1] = v.y;
            to[2] = v.z;
            to[3] = v.w;
            if (v.x != 0.f || v.y != 0.f || v.z != 0.f || v.w != 0.f) from[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < kFoldRows * C; i += kTB) {
            const int r = i % kFoldRows, c = i / kFoldRows;
            const float v = r < n ? rows[r * (cp + 1) + c] : 0.f;
            if (v != 0.f) L64[(size_t)c * nvox + k0 + r] += (double)v;
        }
        __syncthreads();
    }
}

// the gradient tile is padded like the grid the flights walk; its halo receives nothing in valid
// use, and what a replay that left the forward's path added there is dropped
__global__ void k_fold_grad(float* __restrict__ gacc, double* __restrict__ g64, const Geo g) {
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < g.npad; q += gridDim.x * blockDim.x) {
        const float v = gacc[q];
        if (v != 0.f) {
            int k;
            if (interior_lin(g, q, k)) g64[k] += (double)v;
            gacc[q] = 0.f;
        }
    }
}

// dynamic shared memory of a transport block: the warps' photon stacks, the forward's tallies
// and the classic estimate's scratch
template <int MODE>
constexpr size_t smem_bytes() {
    constexpr bool REPLAY = MODE >= 2;
    constexpr bool CLASSIC = MODE == kFwdClassic || MODE == kPass1C || MODE == kPass2C;
    return (size_t)(kTB / 32) * Rec<MODE>::NW * kSlots * sizeof(uint32_t) +
           (REPLAY ? 0 : (size_t)kTB * 15 * sizeof(uint32_t)) +
           (CLASSIC ? (size_t)(kTB / 32) * kClassicWords * sizeof(uint32_t) : 0);
}

// the score kernel's: the warps' flight queues and entry strips
template <int K>
constexpr size_t score_smem() {
    return (size_t)kTransportWarps * score_words<K>() * sizeof(uint32_t);
}

template <typename K>
int occupancy(K kern, size_t smem, int blocks = 3, int threads = kTB) {
    int n = 0;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    {   // shared-memory carveout: enough for the blocks of the kernel's register budget, the rest of the
        // SM's 256 KB to L1, which caches the extinction grid the walks fetch
        const size_t need = blocks * (smem + 1024);
        const int pct = (int)std::min<size_t>(100, (need * 100 + 228 * 1024 - 1) / (228 * 1024));
        cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
    }
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem) != cudaSuccess || n < 1) n = 1;
    return n;
}

template <int DT, int MODE, bool TWO, int TRIP = 0>
cudaError_t launch_mode(const TransportArgs& a, int blocks, cudaStream_t st) {
    if constexpr (TRIP != 0) {  // a variant of the autotuner: the default's carveout (set by occupancy())
        static const int once = occupancy(k_transport<DT, MODE, TWO, TRIP>, smem_bytes<MODE>());
        (void)once;
    }
    k_transport<DT, MODE, TWO, TRIP><<<blocks, kTB, smem_bytes<MODE>(), st>>>(a);
    return cudaGetLastError();
}

// Trip-length variants of the FP32-grid pass-2 kernel, for the autotuner
template <int MODE, bool TWO>
cudaError_t launch_trip(const TransportArgs& a, int trip, int blocks, cudaStream_t st) {
    switch (trip) {
        case 4: return launch_mode<0, MODE, TWO, 4>(a, blocks, st);
        case 8: return launch_mode<0, MODE, TWO, 8>(a, blocks, st);
        case 10: return launch_mode<0, MODE, TWO, 10>(a, blocks, st);
        default: return launch_mode<0, MODE, TWO>(a, blocks, st);
    }
}

template <int DT, bool TWO, int TRIP>
cudaError_t launch_forward_t(const TransportArgs& a, int blocks, cudaStream_t st) {
    if constexpr (TRIP != kForwardTrip) {  // the default's attributes are set by occupancy()
        static const int once = occupancy(k_forward<DT, TWO, TRIP>, forward_smem(), kMinBlocksForward, kFT);
        (void)once;
    }
    k_forward<DT, TWO, TRIP><<<blocks, kFT, forward_smem(), st>>>(a);
    return cudaGetLastError();
}

// The forward of the voxel estimator; FP32 grids have the trip-length variants of the autotuner.
template <int DT, bool TWO>
cudaError_t launch_forward(const TransportArgs& a, int trip, int blocks, cudaStream_t st) {
    if constexpr (DT == 0) {
        switch (trip) {
            case 8: return launch_forward_t<0, TWO, 8>(a, blocks, st);
            case 10: return launch_forward_t<0, TWO, 10>(a, blocks, st);
            case 12: return launch_forward_t<0, TWO, 12>(a, blocks, st);
            case 16: return launch_forward_t<0, TWO, 16>(a, blocks, st);
            default: break;
        }
    }
    return launch_forward_t<DT, TWO, kForwardTrip>(a, blocks, st);
}

template <int DT, bool TWO>
int occupancy_mode(int mode) {
    switch (mode) {
        case kFwdVoxel: return occupancy(k_forward<DT, TWO, kForwardTrip>, forward_smem(), kMinBlocksForward, kFT);
        case kFwdClassic: return occupancy(k_transport<DT, kFwdClassic, TWO>, smem_bytes<kFwdClassic>());
        case kPass2: return occupancy(k_transport<DT, kPass2, TWO>, smem_bytes<kPass2>());
        case kScore: return occupancy(k_score<DT, TWO, kScoreTrip>, score_smem<kScoreTrip>(), kMinBlocksScore, kFT);
        case kPass1C: return occupancy(k_transport<DT, kPass1C, TWO>, smem_bytes<kPass1C>());
        case kPass2C: return occupancy(k_transport<DT, kPass2C, TWO>, smem_bytes<kPass2C>());
        default: return occupancy(k_transport<DT, kPass1, TWO>, smem_bytes<kPass1>());
    }
}

template <int DT, bool TWO>
cudaError_t launch_dt(const TransportArgs& a, int mode, int trip, int blocks, cudaStream_t st) {
    if constexpr (DT == 0) {
        if (trip > 0 && mode == kPass2) return launch_trip<kPass2, TWO>(a, trip, blocks, st);
    }
    switch (mode) {
        case kFwdVoxel: return launch_forward<DT, TWO>(a, trip, blocks, st);
        case kFwdClassic: return launch_mode<DT, kFwdClassic, TWO>(a, blocks, st);
        case kPass2: return launch_mode<DT, kPass2, TWO>(a, blocks, st);
        case kPass1C: return launch_mode<DT, kPass1C, TWO>(a, blocks, st);
        case kPass2C: return launch_mode<DT, kPass2C, TWO>(a, blocks, st);
        default: return launch_mode<DT, kPass1, TWO>(a, blocks, st);
    }
}

template <bool TWO>
cudaError_t launch_species(const TransportArgs& a, int dtype, int mode, int trip, int blocks, cudaStream_t st) {
    return dtype == 0 ? launch_dt<0, TWO>(a, mode, trip, blocks, st)
                      : (dtype == 1 ? launch_dt<1, TWO>(a, mode, trip, blocks, st)
                                    : launch_dt<2, TWO>(a, mode, trip, blocks, st));
}

// The batched form: FP32 grid, one species, the modes of the full gradient with stored events.
// Function attributes (shared memory, carveout) are set by batch_occupancy() before any launch,
// outside a stream capture.
template <int MODE, int TRIP = 0>
cudaError_t launch_batch_mode(const TransportArgs* table, int n, int blocks, cudaStream_t st) {
    k_transport_batch<0, MODE, false, TRIP><<<blocks, kTB, smem_bytes<MODE>(), st>>>(table, n);
    return cudaGetLastError();
}

template <int MODE, int TRIP = 0>
int batch_occupancy() {
    return occupancy(k_transport_batch<0, MODE, false, TRIP>, smem_bytes<MODE>());
}

}  // namespace

cudaError_t launch_transport_batch(const TransportArgs* table, int n, int mode, int trip, int blocks,
                                   cudaStream_t st) {
    switch (mode) {
        case kFwdVoxel:
            switch (trip) {
                case 12: k_forward_batch<12><<<blocks, kFT, forward_smem(), st>>>(table, n); break;
                case 10: k_forward_batch<10><<<blocks, kFT, forward_smem(), st>>>(table, n); break;
                case 16: k_forward_batch<16><<<blocks, kFT, forward_smem(), st>>>(table, n); break;
                default: k_forward_batch<kForwardTrip><<<blocks, kFT, forward_smem(), st>>>(table, n);
            }
            return cudaGetLastError();
        case kPass2: return launch_batch_mode<kPass2>(table, n, blocks, st);
        case kPass1: return launch_batch_mode<kPass1>(table, n, blocks, st);
        default: return cudaErrorInvalidValue;
    }
}

int transport_batch_blocks_per_sm(int mode) {
    static int occ[7] = {0, 0, 0, 0, 0, 0, 0};
    static bool ready = false;
    if (!ready) {  // every instantiation's attributes, once; the default trips give the occupancy
        occ[kFwdVoxel] = occupancy(k_forward_batch<kForwardTrip>, forward_smem(), kMinBlocksForward, kFT);
        occupancy(k_forward_batch<12>, forward_smem(), kMinBlocksForward, kFT);
        occupancy(k_forward_batch<10>, forward_smem(), kMinBlocksForward, kFT);
        occupancy(k_forward_batch<16>, forward_smem(), kMinBlocksForward, kFT);
        occ[kScore] = occupancy(k_score_batch<kScoreTrip>, score_smem<kScoreTrip>(), kMinBlocksScore, kFT);
        occupancy(k_score_batch<4>, score_smem<4>(), kMinBlocksScore, kFT);
        occupancy(k_score_batch<8>, score_smem<8>(), kMinBlocksScore, kFT);
        occupancy(k_score_batch<10>, score_smem<10>(), kMinBlocksScore, kFT);
        occ[kPass2] = batch_occupancy<kPass2>();
        occ[kPass1] = batch_occupancy<kPass1>();
        ready = true;
    }
    return mode >= 0 && mode < 7 && occ[mode] > 0 ? occ[mode] : 1;
}

cudaError_t launch_score_batch(const TransportArgs* table, int n, int trip, int blocks, cudaStream_t st) {
    switch (trip) {
        case 4: k_score_batch<4><<<blocks, kFT, score_smem<4>(), st>>>(table, n); break;
        case 8: k_score_batch<8><<<blocks, kFT, score_smem<8>(), st>>>(table, n); break;
        case 10: k_score_batch<10><<<blocks, kFT, score_smem<10>(), st>>>(table, n); break;
        default: k_score_batch<kScoreTrip><<<blocks, kFT, score_smem<kScoreTrip>(), st>>>(table, n);
    }
    return cudaGetLastError();
}

int transport_blocks_per_sm(int dtype, int mode, bool two) {
    static int cache[2][3][7] = {{{0}}};
    int& c = cache[two ? 1 : 0][dtype][mode];
    if (c) return c;
    if (two)
        c = dtype == 0 ? occupancy_mode<0, true>(mode)
                       : (dtype == 1 ? occupancy_mode<1, true>(mode) : occupancy_mode<2, true>(mode));
    else
        c = dtype == 0 ? occupancy_mode<0, false>(mode)
                       : (dtype == 1 ? occupancy_mode<1, false>(mode) : occupancy_mode<2, false>(mode));
    return c;
}

cudaError_t launch_transport(const mst_grid* g, const TransportArgs& a, int dtype, int mode, int blocks,
                             cudaStream_t st) {
    const int trip = g->wf_trip[mode];  // the handle's wavefront setting (0: the kernel's default)
    return a.beta_air ? launch_species<true>(a, dtype, mode, trip, blocks, st)
                      : launch_species<false>(a, dtype, mode, trip, blocks, st);
}

cudaError_t launch_score_list(const mst_grid* g, uint32_t n, bool stored, cudaStream_t st) {
    const unsigned long long cap = stored ? g->ev_cap : 0ull;
    cudaError_t e = cudaMemsetAsync(g->score_cnt, 0, sizeof(unsigned) * (2 * kScoreBins + 1), st);
    if (e != cudaSuccess) return e;
    const unsigned blocks = (n + kScoreTile - 1) / kScoreTile;
    if (blocks == 0u) return cudaSuccess;
    k_score_hist<<<blocks, kTB, 0, st>>>(g->wbuf, g->nevbuf, n, g->score_cnt, g->ev_count, cap);
    k_score_scatter<<<blocks, kTB, 0, st>>>(g->wbuf, g->nevbuf, n, g->score_cnt, g->score_cnt + kScoreBins,
                                            g->score_cnt + 2 * kScoreBins, g->plist, g->ev_count, cap);
    return cudaGetLastError();
}

namespace {

template <int DT, bool TWO, int K>
cudaError_t launch_score_k(const TransportArgs& a, int blocks, cudaStream_t st) {
    if constexpr (K != kScoreTrip) {  // the default's attributes are set by occupancy()
        static const int once = occupancy(k_score<DT, TWO, K>, score_smem<K>(), kMinBlocksScore, kFT);
        (void)once;
    }
    k_score<DT, TWO, K><<<blocks, kFT, score_smem<K>(), st>>>(a);
    return cudaGetLastError();
}

template <bool TWO>
cudaError_t launch_score_dt(const TransportArgs& a, int dtype, int trip, int blocks, cudaStream_t st) {
    if (dtype == 1) return launch_score_k<1, TWO, kScoreTrip>(a, blocks, st);
    if (dtype == 2) return launch_score_k<2, TWO, kScoreTrip>(a, blocks, st);
    switch (trip) {
        case 4: return launch_score_k<0, TWO, 4>(a, blocks, st);
        case 8: return launch_score_k<0, TWO, 8>(a, blocks, st);
        case 10: return launch_score_k<0, TWO, 10>(a, blocks, st);
        default: return launch_score_k<0, TWO, kScoreTrip>(a, blocks, st);
    }
}

}  // namespace

cudaError_t launch_score(const mst_grid* g, const TransportArgs& a, int dtype, int blocks, cudaStream_t st) {
    const int trip = g->wf_trip[kScore];
    return a.beta_air ? launch_score_dt<true>(a, dtype, trip, blocks, st)
                      : launch_score_dt<false>(a, dtype, trip, blocks, st);
}

cudaError_t launch_fold_L(const mst_grid* g, cudaStream_t st) {
    const int nb = (g->geo.nvox + kFoldRows - 1) / kFoldRows;
    const size_t smem = sizeof(float) * kFoldRows * (g->cp + 1);
    k_fold_L<<<nb < 4096 ? nb : 4096, kTB, smem, st>>>(g->Lacc, g->L64, g->geo.nvox, g->n_cams, g->cp);
    return cudaGetLastError();
}

cudaError_t launch_fold_grad(const mst_grid* g, cudaStream_t st) {
    const int nb = (g->geo.npad + 255) / 256;
    k_fold_grad<<<nb < 4096 ? nb : 4096, 256, 0, st>>>(g->gacc, g->g64, g->geo);
    return cudaGetLastError();
}

}  // namespace mst
