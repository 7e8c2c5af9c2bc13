"""How a ray on the padded grid ends, compiled for the host from the header that the kernels include: the
walk and the ending rule of the backward paths over lattice directions and starts, where faces of two or
three axes are met at once."""
import importlib.util
import os
import subprocess

import pytest

from tests.conftest import ROOT

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#include "mst_dev.cuh"
using namespace mst;

int main() {
    Geo g{};
    g.nx = 5, g.ny = 4, g.nz = 6;
    g.max_steps = g.nx + g.ny + g.nz + 8;
    g.p0 = g.nx + 2 * kHalo;
    g.p01 = g.p0 * (g.ny + 2 * kHalo);
    g.npad = g.p01 * (g.nz + 2 * kHalo);
    const float hs[2][3] = {{1.f, 1.f, 1.f}, {50.f, 40.f, 60.f}};
    long rays = 0, zero = 0, outside = 0, astray = 0, endless = 0;
    for (auto& h : hs)
        for (float ext : {0.f, 1e-4f}) {
            g.hx = h[0], g.hy = h[1], g.hz = h[2];
            std::vector<float> beta(g.npad, INFINITY);
            for (int z = 0; z < g.nz; ++z)
                for (int y = 0; y < g.ny; ++y)
                    for (int x = 0; x < g.nx; ++x) beta[pad_index(g, x, y, z)] = ext;
            for (int dir = 0; dir < 343; ++dir)
                for (int off = 0; off < 125; ++off)
                    for (int at = 0; at < g.nx * g.ny * g.nz; at += 7)
                        for (bool flight : {false, true}) {
                            // along the diagonals of voxels, so that every start offset that is the same
                            // fraction of each axis ties
                            const float vx = (dir % 7 - 3) * h[0], vy = (dir / 7 % 7 - 3) * h[1], vz = (dir / 49 - 3) * h[2];
                            const float n = std::sqrt(vx * vx + vy * vy + vz * vz);
                            if (n == 0.f) continue;
                            const float3 d = make_float3(vx / n, vy / n, vz / n);
                            const float3 p = make_float3(off % 5 * 0.25f * h[0], off / 5 % 5 * 0.25f * h[1], off / 25 * 0.25f * h[2]);
                            const int ix = at % g.nx, iy = at / g.nx % g.ny, iz = at / (g.nx * g.ny);
                            PadWalk w = pad_walk(g, p, d, ix, iy, iz);
                            float tau = 1e30f, bn = beta[w.lin];
                            int last = -1;
                            ++rays;
                            for (int k = 0;; ++k) {
                                bool px, py;
                                int next;
                                const float b = bn, m = w.face(px, py, next);
                                if (next < 0 || next >= g.npad) { ++outside; break; }  // a load past the array
                                bn = beta[next];
                                if (std::isinf(b) && m == 0.f) ++zero;
                                const float bs = b * m;
                                if (ray_ends(flight, tau, b, bs)) {
                                    // the first halo voxel after the last one of the grid
                                    if (!std::isinf(b) || last < 0 || std::isinf(beta[last])) ++astray;
                                    break;
                                }
                                if (k > g.max_steps) { ++endless; break; }
                                tau -= bs;
                                last = w.lin;
                                w.cross(m, px, py, next);
                            }
                        }
        }
    std::printf("%ld %ld %ld %ld %ld\n", rays, zero, outside, astray, endless);
}
"""


def test_rays_end_in_the_first_halo_voxel(tmp_path):
    spec = importlib.util.spec_from_file_location("mst_cuda_build", os.path.join(ROOT, "paper_1512_02110_gb300", "build.py"))
    build = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(build)
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "walk.cu", tmp_path / "walk"
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-Xcompiler", "-ffp-contract=off", "-I", build.CSRC,
                    str(src), "-o", str(exe)] + build.ARCH, check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rays, zero, outside, astray, endless = map(int, out.split())
    assert rays > 10**6 and zero > 1000  # first halo voxels met on an edge: no distance in them
    assert (outside, astray, endless) == (0, 0, 0)
