"""Workloads of the library as its users run them: forward renders, renders with a gradient, the
paper's inner loop on a fixed in-scatter field, ray geometry on its own, backward Monte Carlo and
batches of uneven scenes.

A case is a dict of plain values. `prepare` builds what a program has in hand before a call (the
extinction field on the device, the grid handle, measured images), `run` makes one call through the
package's public API, `exact` repeats the deterministic ones in 64-bit torch. Fields, cameras and
measurements are synthetic and follow from the seed alone.

Sizes are those of the repository's own configurations: grids of 16^3 to 96^3 (80 x 80 x 120 for
the haze of the paper), 3 to 36 cameras of 32^2 to 128^2 pixels, 1e5 to 1e8 photons.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1512_02110_gb300 as mst

KM = 1e-3  # 1/km in 1/m

BASE = dict(field="cumulus", nx=64, ny=64, nz=64, voxel=20.0, cams=9, px=128, photons=0, albedo=0.999, g=0.85,
            zenith=45.0, dtype="f32", estimator="voxel", grad="full", eta=0.0, paths=0, scenes=0)


def _case(name, op, **kw):
    return dict(BASE, name=name, op=op, **kw)


def listed():
    return [
        # the smallest call in use: one quick-look render of a 16^3 scene, where launches and the
        # longest photon path count more than throughput
        _case("render_small", "render", field="blobs", nx=16, ny=16, nz=16, voxel=50.0, cams=5, px=32, photons=100_000,
              albedo=0.99, zenith=30.0),
        # one gradient step of a small reconstruction: a chain of some thirty short launches
        _case("grad_small", "grad", field="blobs", nx=16, ny=16, nz=16, voxel=50.0, cams=5, px=32, photons=100_000,
              albedo=0.99, zenith=30.0),
        # a forward render that refreshes the in-scatter field between inner loops (L returned)
        _case("render_64", "render", photons=20_000_000),
        # gradient of the 32^3 differentiable configuration
        _case("grad_32", "grad", field="blobs", nx=32, ny=32, nz=32, voxel=40.0, px=64, photons=10_000_000),
        # the headline: one reconstruction iteration at 64^3, nine in-situ cameras, 1e8 photons
        _case("grad_64", "grad", photons=100_000_000),
        # the same scene with the extinction grid kept in 16 bits, and a regulariser
        _case("grad_64_bf16", "grad", photons=10_000_000, dtype="bf16", eta=10.0),
        # aerosol and air together under 36 ground cameras: the paper's haze on its grid
        _case("grad_haze", "grad", field="haze", nx=80, ny=80, nz=120, voxel=625.0, cams=36, px=64, photons=10_000_000,
              albedo=0.9, g=0.7),
        # the comparison estimator (a shadow ray from every event to every camera)
        _case("classic_64", "grad", photons=500_000, estimator="classic"),
        # the paper's inner loop: loss and gradient with the in-scatter field held fixed (no photons)
        _case("inner_64", "inner"),
        # ray geometry alone on an odd-sized grid with cameras of unlike sizes: transmittance to
        # every camera, and images of a given field
        _case("views_odd", "views", nx=95, ny=77, nz=61, cams=11, px=97),
        # backward paths from every pixel, the check of the forward model
        _case("bmc_64", "bmc", paths=16),
        # scenes of uneven size in one batch call
        _case("batch_uneven", "batch", nx=96, ny=96, nz=96, cams=12, px=128, photons=8_000_000, scenes=6),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges."""
    op = rng.choice(["render", "grad", "grad", "grad", "inner", "views", "bmc", "batch"])
    c = dict(BASE, op=op, field=rng.choice(["blobs", "cumulus", "cumulus", "haze"]), albedo=round(rng.uniform(0.99, 0.999), 4),
             g=round(rng.uniform(0.75, 0.9), 3), zenith=round(rng.uniform(0.0, 60.0), 1))
    c["nx"], c["ny"], c["nz"] = (round(_log(rng, 16, 96)) for _ in range(3))
    c["cams"], c["px"], c["voxel"] = rng.randint(3, 12), round(_log(rng, 32, 128)), rng.choice([20.0, 40.0, 50.0])
    if c["field"] == "haze":
        c.update(voxel=625.0, cams=rng.randint(9, 36), px=round(_log(rng, 32, 64)), albedo=0.9, g=0.7)
    if op in ("render", "grad"):
        c["photons"] = round(_log(rng, 1e5, 2e7))
        c["dtype"] = rng.choice(["f32", "f32", "f16", "bf16"])
    if op == "grad":
        kind = rng.choice(["full", "full", "surrogate", "classic"])
        if kind == "classic":
            c.update(estimator="classic", photons=round(_log(rng, 5e4, 5e5)))
        elif kind == "surrogate":
            c["grad"] = "surrogate"
        c["eta"] = rng.choice([0.0, 10.0])
    if op in ("bmc", "batch") and c["field"] == "haze":  # one species, both
        c.update(field="cumulus", voxel=20.0, cams=rng.randint(3, 12))
    if op == "bmc":
        c["paths"] = round(_log(rng, 4, 32))
    if op == "batch":
        c.update(scenes=rng.randint(2, 6), photons=round(_log(rng, 1e5, 8e6)))
    return c


# ---------------------------------------------------------------------------------------------
# inputs


def _smooth(rng, shape, power):
    """Gaussian random field, amplitude |k|^power, unit variance ([nz][ny][nx])."""
    k = np.meshgrid(*[np.fft.fftfreq(n) for n in shape], indexing="ij")
    kk = np.sqrt(sum(v * v for v in k))
    kk.flat[0] = 1.0
    amp = kk ** power
    amp.flat[0] = 0.0
    f = np.real(np.fft.ifftn(np.fft.fftn(rng.standard_normal(shape)) * amp))
    return f / f.std()


def _blobs(rng, shape, n, sigma):
    """Sum of n Gaussian blobs in unit coordinates, maximum 1; sigma: (z, y, x) ranges."""
    z, y, x = np.meshgrid(*[(np.arange(m) + 0.5) / m for m in shape], indexing="ij")
    f = np.zeros(shape)
    for _ in range(n):
        c = rng.uniform(0.2, 0.8, 3)
        s = [rng.uniform(*v) for v in sigma]
        f += np.exp(-0.5 * (((z - c[0]) / s[0]) ** 2 + ((y - c[1]) / s[1]) ** 2 + ((x - c[2]) / s[2]) ** 2))
    return f / f.max()


def _field(case, rng):
    """Extinction [nz][ny][nx] in 1/m, and the air's or None."""
    shape = (case["nz"], case["ny"], case["nx"])
    if case["field"] == "blobs":  # three blobs over a thin background
        return 20 * KM * _blobs(rng, shape, 3, [(0.12, 0.25)] * 3) + 0.01 * KM, None
    if case["field"] == "cumulus":  # k^-5/3 cloud, fraction 0.3, clear air between
        f = _smooth(rng, shape, -11.0 / 6.0)
        thr = np.quantile(f, 0.7)
        return np.where(f > thr, 80 * KM * (f - thr) / (f.max() - thr), 0.0), None
    # haze: blobs wide across and shallow in altitude over a background, and molecular air at 550 nm
    f = 0.2 * KM * _blobs(rng, shape, 4, [(0.05, 0.12), (0.08, 0.18), (0.08, 0.18)]) + 0.005 * KM
    z = (np.arange(shape[0]) + 0.5) * 10000.0 / shape[0]
    return f, np.broadcast_to(0.0116 * KM * np.exp(-z / 8000.0)[:, None, None], shape)


def _size(case):
    v = case["voxel"]
    return (v, v, 10000.0 / case["nz"]) if case["field"] == "haze" else (v, v, v)


def _cameras(case, rng, beta):
    """Cameras looking up from the ground on a jittered lattice; in a cloud, every fourth one raised
    into it (in situ). Image sizes differ from camera to camera when px is odd."""
    h, n = _size(case), case["cams"]
    ext = [case["nx"] * h[0], case["ny"] * h[1]]
    m = math.ceil(math.sqrt(n))
    pos = []
    for c in range(n):
        x, y = ((c % m + rng.uniform(0.3, 0.7)) / m * ext[0], (c // m + rng.uniform(0.3, 0.7)) / m * ext[1])
        z = 1.0
        if case["field"] == "cumulus" and c % 4 == 0:
            col = np.nonzero(beta[:, min(int(y / h[1]), case["ny"] - 1), min(int(x / h[0]), case["nx"] - 1)])[0]
            z = (col[0] + 0.4) * h[2] if col.size else z
        pos.append((x, y, z))
    odd = case["px"] % 2 == 1
    w = np.array([case["px"] - (5 * c if odd else 0) % (case["px"] // 2) for c in range(n)])
    hgt = np.array([case["px"] - (3 * c if odd else 0) % (case["px"] // 2) for c in range(n)])
    fov = math.radians(150.0 if case["field"] == "haze" else 60.0)
    return dict(cam_pos=np.array(pos), cam_rot=np.tile(np.eye(3).ravel(), (n, 1)), cam_w=w, cam_h=hgt,
                cam_fov=np.full(n, fov), n_rays=10)


def _measured(rng, cams):
    """Measured images: a slow pattern per camera and pixel noise, of the sky's order of brightness."""
    out = []
    for w, h in zip(cams["cam_w"], cams["cam_h"]):
        y, x = np.meshgrid(np.linspace(0, 1, h), np.linspace(0, 1, w), indexing="ij")
        f = 0.08 + 0.04 * np.sin(6.3 * (x * rng.uniform(0.2, 1) + rng.random())) * np.cos(6.3 * y * rng.uniform(0.2, 1))
        out.append((f * (1 + 0.01 * rng.standard_normal(f.shape))).ravel())
    return np.concatenate(out)


def _dev(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype).reshape(-1)


def _scene(case, seed):
    """Everything of one scene on the host: arrays and the arguments of the handle."""
    rng = np.random.default_rng(seed)
    beta, air = _field(case, rng)
    cams = _cameras(case, rng, beta)
    s = dict(beta=beta, air=air, cams=cams, args=dict(shape=(case["nx"], case["ny"], case["nz"]), h=_size(case),
                                                      origin=(0.0, 0.0, 0.0), **cams))
    if case["op"] in ("grad", "inner", "batch"):
        s["meas"] = _measured(rng, cams)
    if case["op"] in ("inner", "views"):  # in-scatter per camera: proportional to the extinction, slowly varying
        j = np.stack([np.exp(0.3 * _smooth(rng, beta.shape, -2.0)) for _ in range(3)])
        s["L"] = np.stack([beta * j[c % 3] * (0.5 + c / case["cams"]) for c in range(case["cams"])]) * 1e3
        s["beta_now"] = beta * np.exp(0.2 * _smooth(rng, beta.shape, -2.0))
    return s


def _params(case, seed, photons):
    return mst.make_params(albedo=case["albedo"], g=case["g"], sun_zenith=math.radians(case["zenith"]),
                           n_photons=max(photons, 1), seed=seed % (1 << 30) + 3, estimator=case["estimator"],
                           grid_dtype=case["dtype"], grad_mode=case["grad"], reg_eta=case["eta"])


def _batch_cases(case):
    """The scenes of a batch: sizes falling from the case's grid to a quarter of it, alternating fields."""
    n, out = case["scenes"], []
    for i in range(n):
        f = 1.0 - 0.75 * i / n
        out.append(dict(case, field="blobs" if i % 2 else "cumulus", nx=max(8, round(case["nx"] * f)),
                        ny=max(8, round(case["ny"] * f)), nz=max(8, round(case["nz"] * f)),
                        cams=max(3, round(case["cams"] * f)), px=case["px"] if i % 2 else max(16, case["px"] // 2),
                        photons=max(1000, round(case["photons"] / (1 + i % 3)))))
    return out


def prepare(case, seed):
    if case["op"] == "batch":
        parts = [prepare(dict(c, op="grad", scenes=0), seed + 1000 * i) for i, c in enumerate(_batch_cases(case))]
        return dict(case=case, parts=parts, batch=mst.Batch([p["grid"] for p in parts]))
    s = _scene(case, seed)
    st = dict(case=case, grid=mst.Grid(**s["args"]), params=_params(case, seed, case["photons"]),
              beta=_dev(s["beta"], torch.float32))
    if s["air"] is not None and case["op"] not in ("inner", "views"):
        st["grid"].set_air(_dev(s["air"], torch.float32), 1.0)
    if "meas" in s:
        st["meas"] = _dev(s["meas"], torch.float64)
    if "L" in s:
        st["L"] = _dev(s["L"], torch.float64)
        st["beta_now"] = _dev(s["beta_now"], torch.float32)
    return st


def run(state):
    case, op = state["case"], state["case"]["op"]
    if op == "batch":
        p = state["parts"]
        return state["batch"].render_grad([q["beta"] for q in p], [q["params"] for q in p], [q["meas"] for q in p],
                                          images=True)
    g = state["grid"]
    if op == "render":
        return g.render(state["beta"], state["params"], images=True, L=True)
    if op == "grad":
        return g.render_grad(state["beta"], state["params"], state["meas"])
    if op == "inner":
        return g.surrogate_grad(state["beta_now"], state["L"], state["beta"], state["params"], state["meas"])
    if op == "views":
        return dict(T=g.transmittance(state["beta"]), images=g.form_images(state["beta"], state["L"]))
    return g.render_bmc(state["beta"], state["params"], case["paths"])


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without


def _photon_work(case):
    """Voxel segments and events per photon, roughly: a photon crosses about a third of the grid's
    three extents; events follow the field's mean optical depth."""
    seg = 0.36 * (case["nx"] + case["ny"] + case["nz"])
    per = {"cumulus": 3.9 * case["nz"] * case["voxel"] / 1280.0, "blobs": 3.0 * case["nz"] * case["voxel"] / 800.0, "haze": 0.3}
    return seg, per[case["field"]]


def _ray_segments(case):
    """Voxel segments of one pass over the lines of sight, and of one over the pixel rays."""
    nvox, side = case["nx"] * case["ny"] * case["nz"], (case["nx"] + case["ny"] + case["nz"]) / 3
    return case["cams"] * nvox * 0.8 * side, case["cams"] * case["px"] ** 2 * 10 * 1.3 * side


def work(case):
    """Bytes of the inputs and outputs, each once; operations: 15 per voxel segment of a photon's flight, 35 per
    event and 27 per event and camera, and 6 per segment of a camera ray or line of sight."""
    if case["op"] == "batch":
        parts = [work(dict(c, op="grad", scenes=0)) for c in _batch_cases(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    nvox, C, npix = case["nx"] * case["ny"] * case["nz"], case["cams"], case["cams"] * case["px"] ** 2
    seg, ev = _photon_work(case)
    los, pix = _ray_segments(case)
    n, op = case["photons"], case["op"]
    if op == "render":
        return {"bytes": 4 * nvox + 8 * npix + 8 * C * nvox, "flops": n * (15 * seg + ev * (35 + 27 * C)) + 6 * (los + pix)}
    if op == "grad":
        rays = 12 * (los + pix) if case["estimator"] == "voxel" else n * ev * C * 45 * seg
        replay = n * (10 * seg + ev * 27 * C) if case["grad"] == "full" else 0
        return {"bytes": 4 * nvox * (2 if case["field"] == "haze" else 1) + 8 * nvox + 16 * npix,
                "flops": n * (15 * seg + ev * (35 + 27 * C)) + replay + rays}
    if op == "inner":
        return {"bytes": 8 * nvox + 8 * C * nvox + 8 * nvox + 16 * npix, "flops": 12 * (los + pix)}
    if op == "views":
        return {"bytes": 4 * nvox + 4 * C * nvox + 8 * C * nvox + 8 * npix, "flops": 6 * (los + pix)}
    return {"bytes": 4 * nvox + 16 * npix, "flops": npix * case["paths"] * (30 * seg + ev * 62)}


# ---------------------------------------------------------------------------------------------
# 64-bit references of the deterministic calls


def _walk(shape, h, p, d, end, visit):
    """Walks rays from points p along unit directions d ([n, 3], inside the grid) to the distance
    `end` or the grid's boundary; visit(rays, voxel, length) once per lockstep of the rays left."""
    dev = p.device
    n3 = torch.tensor(shape, device=dev)
    hh = torch.tensor(h, dtype=torch.float64, device=dev)
    i = torch.minimum(torch.clamp((p / hh).floor().long(), min=0), n3 - 1)
    rays, t = torch.arange(len(p), device=dev), torch.zeros(len(p), dtype=torch.float64, device=dev)
    step = torch.sign(d).long()
    while len(rays):
        face = ((i + (step > 0)) * hh - p) / d
        face = torch.where(step == 0, torch.full_like(face, math.inf), face)
        tn, axis = face.min(1)
        tn = torch.minimum(torch.maximum(tn, t), end)
        visit(rays, i[:, 0] + shape[0] * (i[:, 1] + shape[1] * i[:, 2]), tn - t)
        i = i + torch.nn.functional.one_hot(axis, 3) * step
        keep = (tn < end) & ((i >= 0) & (i < n3)).all(1)
        rays, p, d, end, i, step, t = (v[keep] for v in (rays, p, d, end, i, step, tn))


def _radical_inverse(base, k):
    f, r = 1.0, 0.0
    while k:
        f /= base
        r += f * (k % base)
        k //= base
    return r


class _Rays:
    """Lines of sight and pixel rays of a scene in 64 bits, on the device for their number."""

    def __init__(self, s):
        self.shape, self.h, self.cams = s["args"]["shape"], s["args"]["h"], s["cams"]
        self.C, self.nvox = len(self.cams["cam_pos"]), int(np.prod(self.shape))
        self.pos = torch.tensor(self.cams["cam_pos"], dtype=torch.float64, device="cuda")
        k = torch.arange(self.nvox, device="cuda")
        ijk = torch.stack([k % self.shape[0], k // self.shape[0] % self.shape[1], k // (self.shape[0] * self.shape[1])], 1)
        self.centres = (ijk + 0.5) * torch.tensor(self.h, dtype=torch.float64, device="cuda")

    def los(self, c, visit):
        v = self.pos[c] - self.centres
        dist = v.norm(dim=1)
        _walk(self.shape, self.h, self.centres, v / dist[:, None], dist, visit)

    def pixels(self, c, visit):
        """visit(pixel of the camera's block, voxel, length)"""
        w, hgt, n_rays = int(self.cams["cam_w"][c]), int(self.cams["cam_h"][c]), self.cams["n_rays"]
        tx = math.tan(0.5 * self.cams["cam_fov"][c])
        q = torch.arange(w * hgt, device="cuda")
        for r in range(n_rays):
            x = (2 * ((q % w) + _radical_inverse(2, r + 1)) / w - 1).double() * tx
            y = (2 * ((q // w) + _radical_inverse(3, r + 1)) / hgt - 1).double() * (tx * hgt / w)
            d = torch.stack([x, y, torch.ones_like(x)], 1)  # the cameras look up: right x, up y, forward z
            d = d / d.norm(dim=1, keepdim=True)
            _walk(self.shape, self.h, self.pos[c].expand_as(d).contiguous(), d,
                  torch.full((len(q),), math.inf, dtype=torch.float64, device="cuda"), visit)

    def transmittance(self, beta):
        T = torch.zeros(self.C, self.nvox, dtype=torch.float64, device="cuda")
        for c in range(self.C):
            self.los(c, lambda r, k, l: T[c].index_add_(0, r, beta[k] * l))
        return torch.exp(-T)

    def images(self, R):
        scale = 1.0 / (self.cams["n_rays"] * float(np.prod(self.h)))
        out = []
        for c in range(self.C):
            img = torch.zeros(int(self.cams["cam_w"][c] * self.cams["cam_h"][c]), dtype=torch.float64, device="cuda")
            self.pixels(c, lambda r, k, l: img.index_add_(0, r, R[c][k] * l))
            out.append(img * scale)
        return torch.cat(out)


def exact(case, seed):
    """Transmittance, images and the fixed-field gradient in plain 64-bit torch. The Monte-Carlo
    calls have no such value: a photon whose free path ends within rounding of a voxel's face takes
    another path in 64 bits, and what one photon adds is not small beside the result."""
    if case["op"] not in ("inner", "views"):
        return None
    s = _scene(case, seed)
    ray = _Rays(s)
    f32 = lambda a: _dev(a, torch.float32).double()
    L = _dev(s["L"], torch.float64).view(ray.C, ray.nvox)
    if case["op"] == "views":
        T = ray.transmittance(f32(s["beta"]))
        return dict(T=T, images=ray.images(L * T))
    ref, now = f32(s["beta"]), f32(s["beta_now"])
    T = ray.transmittance(now)
    j = torch.where(ref > 0, L / ref.clamp(min=1e-300), torch.zeros_like(L))
    R = j * now * T
    img = ray.images(R)
    res = img - _dev(s["meas"], torch.float64)
    scale = 1.0 / (ray.cams["n_rays"] * float(np.prod(ray.h)))
    grad, off = torch.zeros(ray.nvox, dtype=torch.float64, device="cuda"), 0
    for c in range(ray.C):
        n = int(ray.cams["cam_w"][c] * ray.cams["cam_h"][c])
        q, off = 2 * scale * res[off:off + n], off + n
        b = torch.zeros_like(grad)
        ray.pixels(c, lambda r, k, l: b.index_add_(0, k, q[r] * l))
        grad += j[c] * T[c] * b
        Rb = R[c] * b
        ray.los(c, lambda r, k, l: grad.index_add_(0, k, -Rb[r] * l))
    return dict(loss=(res * res).sum().reshape(1), grad=grad, images=img)
