"""The forward, score and ray kernels at the sizes where their tiles, queues and batches have edges:
single photons and batches that never fill, grids of odd and single-voxel extents (half-empty bricks
of the score's tile), camera counts around the groups of two, four and eight, a sun straight down
(flights along one axis only), sub-pixel ray counts that do not divide a block."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import dev, f32_scene, gpu_hashes, max_rel, need_gpu, record, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    return need_gpu()


def _scene(shape, cams, seed, n_rays=10, px=(8, 6), outside=False):
    rng = np.random.default_rng(seed)
    h = (50.0, 40.0, 60.0)
    beta = rng.uniform(1.0, 15.0, int(np.prod(shape))) * synth.KM
    ext = np.array(shape) * np.array(h)
    pos = np.column_stack([ext[0] * rng.uniform(0.2, 0.8, cams), ext[1] * rng.uniform(0.2, 0.8, cams),
                           np.full(cams, -25.0 if outside else 1.0)])
    c = synth.make_cameras(pos, px[0], px[1], 70.0)
    return f32_scene(synth.make_scene(shape, h, beta, c, n_rays=n_rays))


# (grid, cameras, photons, sun zenith): a launch of one photon; one batch of 32 and one more; rounds
# that drain with fewer than 32 events; several chunks of records per warp
CASES = [((1, 1, 1), 1, 33, 0.6), ((2, 3, 1), 4, 1, 0.0), ((5, 7, 9), 5, 33, 0.0), ((5, 7, 9), 13, 5000, 0.7),
         ((33, 17, 12), 17, 70_001, 0.3), ((16, 16, 16), 9, 400_000, 0.0)]


def _full_gradient(shape, cams, photons, zenith, estimator):
    sc = _scene(shape, cams, 7)
    p = synth.Params(albedo=0.95, g=0.7, sun_zenith=zenith, sun_azimuth=0.4, n_photons=photons, seed=11)
    return sc, p, dict(grad_mode="full", estimator=estimator), np.linspace(0.0, 0.1, sc.n_pix)


@pytest.mark.parametrize("shape,cams,photons,zenith", CASES)
def test_score_of_stored_events_matches_the_replay(m, shape, cams, photons, zenith):
    """The gradient from the stored events (k_forward, k_score) against the one of the replay passes,
    which walk every photon again from its Philox key in a kernel of their own: the same terms in
    another order, so the two agree to the rounding of FP32 sums (1e-5, the bound of the
    repository's other comparison of the two forms)."""
    sc, p, opt, meas = _full_gradient(shape, cams, photons, zenith, "voxel")
    a_grid, b_grid = m.Grid.from_scene(sc), m.Grid.from_scene(sc)
    b_grid.set_replay_memory(0)
    a, b = (g.render_grad(dev(sc.beta, np.float32), m.make_params(p, **opt), dev(meas, np.float64)) for g in (a_grid, b_grid))
    sa, sb = a_grid.stats(), b_grid.stats()
    for k in ("events", "segments", "escaped_n", "traced"):
        assert sa[k] == sb[k], (k, sa[k], sb[k])
    assert sa["lost"] == 0 and sa["traced"] == photons
    assert sa["events_stored"] == sa["events"] and sb["events_stored"] == 0
    ga, gb = a["grad"].cpu().numpy(), b["grad"].cpu().numpy()
    assert np.isfinite(ga).all()
    eg = rel_l2(ga, gb) if np.any(gb) else float(np.abs(ga).max())
    record(f"score_vs_replay[{shape},{cams},{photons}]", grad_rel_l2=eg, events=sa["events"])
    assert eg < 1e-5, eg


@pytest.mark.parametrize("shape,cams,photons,zenith", CASES)
def test_classic_gradient_matches_the_oracle(m, shape, cams, photons, zenith):
    """The classic estimate's gradient against the FP64 oracle on the photons whose paths agree.
    1e-3: the bound of the repository's other gradients against the oracle."""
    sc, p, opt, meas = _full_gradient(shape, cams, photons, zenith, "classic")
    beta, grid = dev(sc.beta, np.float32), m.Grid.from_scene(sc)
    ref_hash = oracle.render(sc, p, want_L=False, hashes=True)["hash"]
    skip = (gpu_hashes(m, grid, beta, m.make_params(p), photons) != ref_hash).astype(np.uint8)
    assert skip.mean() < 2e-3
    skip_dev = dev(skip, np.uint8)
    grid.set_debug(None, skip_dev)
    out = grid.render_grad(beta, m.make_params(p, **opt), dev(meas, np.float64))
    grid.set_debug(None, None)
    ref = oracle.full_grad(sc, p, meas, skip=skip, classic=True)
    assert grid.stats()["lost"] == 0
    eg = rel_l2(out["grad"].cpu().numpy(), ref["grad"])
    el = abs(out["loss"].item() - ref["loss"]) / ref["loss"]
    record(f"classic_gradient[{shape},{cams},{photons}]", grad_rel_l2=eg, loss=el)
    assert eg < 1e-3 and el < 1e-3, (eg, el)


@pytest.mark.parametrize("shape,cams,n_rays,px,outside", [((1, 1, 1), 1, 1, (1, 1), False), ((5, 7, 9), 3, 7, (5, 3), False),
                                                          ((9, 5, 4), 2, 64, (9, 4), True), ((33, 17, 12), 5, 10, (33, 9), True)])
def test_rays_match_the_oracle(m, shape, cams, n_rays, px, outside):
    """Transmittance, images of a given field, and the fixed-field loss and gradient against the FP64
    oracle: FP32 chords leave 1e-6 of a segment, the bounds of the repository's other ray tests
    (2e-6 + 2e-5 max(tau, 1), 1e-4 of an image, 1e-3 of the gradient) hold here too."""
    sc = _scene(shape, cams, 3, n_rays=n_rays, px=px, outside=outside)
    rng = np.random.default_rng(5)
    L = rng.uniform(0.5, 2.0, (cams, sc.nvox)) * sc.beta
    meas = rng.uniform(0.0, 1e-4, sc.n_pix)
    now = (sc.beta * rng.uniform(0.8, 1.2, sc.nvox)).astype(np.float32).astype(np.float64)
    grid, beta = m.Grid.from_scene(sc), dev(sc.beta, np.float32)
    tau, T_ref = oracle.transmittance(sc)
    eT = []
    for T in (grid.transmittance(beta),  # the handle's haloed copy of beta, and the linear one without a handle
              m.transmittance_noalloc(sc.shape, sc.h, sc.origin, sc.cam_pos, sc.cam_rot, sc.cam_w, sc.cam_h, sc.cam_fov, beta)):
        err = np.abs(T.cpu().numpy() - T_ref) / T_ref
        eT.append(float(np.max(err / (2e-5 * np.maximum(tau, 1.0) + 2e-6))))
    img = grid.form_images(beta, dev(L, np.float64).view(cams, -1)).cpu().numpy()
    img_ref = oracle.images(sc, L, T_ref)
    ei = max_rel(img, img_ref, 1e-3 * np.abs(img_ref).max())
    out = grid.surrogate_grad(dev(now, np.float32), dev(L, np.float64).view(cams, -1), beta, m.make_params(synth.Params()),
                              dev(meas, np.float64))
    ref = oracle.surrogate_grad(sc.with_beta(now), L, sc.beta, meas)
    el = abs(out["loss"].item() - ref["loss"]) / ref["loss"]
    eg = rel_l2(out["grad"].cpu().numpy(), ref["grad"])
    record(f"rays[{shape},{n_rays},{px}]", T=eT[0], T_noalloc=eT[1], images=ei, loss=el, grad=eg)
    assert max(eT) <= 1.0 and ei < 1e-4 and el < 1e-4 and eg < 1e-3, (eT, ei, el, eg)


@pytest.mark.parametrize("shape,cams,paths", [((1, 1, 1), 1, 33), ((5, 7, 9), 3, 64), ((33, 17, 12), 5, 200)])
def test_backward_paths_all_end(m, shape, cams, paths):
    """Every backward path ends in a collision or at the grid's boundary: none is abandoned, and a ray
    crosses no more voxels than a straight line through the grid has."""
    sc = _scene(shape, cams, 9)
    grid = m.Grid.from_scene(sc)
    p = synth.Params(albedo=0.95, g=0.7, sun_zenith=0.5, sun_azimuth=0.4, seed=21)
    out = grid.render_bmc(dev(sc.beta, np.float32), m.make_params(p), paths)
    st = grid.stats()
    assert st["lost"] == 0 and st["bmc_paths"] == paths * sc.n_pix and st["bmc_events"] > 0
    # one flight a path and two rays an event
    assert st["bmc_segments"] <= (st["bmc_paths"] + 2 * st["bmc_events"]) * sum(shape)
    assert np.isfinite(out["images"].cpu().numpy()).all()


def test_backward_paths_of_both_kernels(m):
    """A call with few paths walks a path's rays in turn, one with many takes them in trips: the same
    Philox streams, so the first paths of every pixel are the same whichever kernel runs. 64 x 65 x 66 voxels, 10
    paths per resident lane and more for five cameras (one kernel), the first camera alone (the other): its means
    and spreads agree to the rounding of FP64 sums (1e-12)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = -(-10 * sms * 1024 // (5 * 33 * 33)) + 1  # paths a pixel
    sc = _scene((64, 65, 66), 5, 9, px=(33, 33))
    p = m.make_params(synth.Params(albedo=0.95, g=0.7, sun_zenith=0.5, sun_azimuth=0.4, seed=21))
    beta = dev(sc.beta, np.float32)
    grid = m.Grid.from_scene(sc)
    a = grid.render_bmc(beta, p, n)
    st = grid.stats()
    assert st["lost"] == 0 and st["bmc_paths"] == n * sc.n_pix >= 10 * sms * 1024
    first = m.Grid(sc.shape, sc.h, sc.origin, sc.cam_pos[:1], sc.cam_rot[:1], sc.cam_w[:1], sc.cam_h[:1], sc.cam_fov[:1],
                   sc.n_rays)
    c = first.render_bmc(beta, p, n)
    st = first.stats()
    assert st["lost"] == 0 and st["bmc_paths"] == n * 33 * 33 < 10 * sms * 1024
    for k in ("images", "var"):
        x, y = a[k][: 33 * 33].cpu().numpy(), c[k].cpu().numpy()
        assert np.abs(x - y).max() <= 1e-12 * np.abs(x).max(), k


def test_a_new_handle_is_ready_for_any_stream(m):
    """Creation leaves no work in flight: the clears of the handle's buffers (here some 0.3 GB, behind work
    that was queued before) are done when it returns, so that a first call on a stream that does not wait
    for the default one finds R's halo marked and the tiles empty."""
    torch.cuda.synchronize()
    sc = _scene((128, 128, 128), 16, 3, px=(4, 4))
    torch.cuda._sleep(1_000_000)
    grid = m.Grid.from_scene(sc)
    assert torch.cuda.default_stream().query()
    beta = dev(sc.beta, np.float32)
    L = dev(np.ones((16, sc.nvox)), np.float64)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()  # (torch's streams do not block on the legacy one)
    fresh = m.Grid.from_scene(sc)
    with torch.cuda.stream(side):
        img = fresh.form_images(beta, L)
    side.synchronize()
    assert torch.equal(img, grid.form_images(beta, L))


def test_thin_grids_hold_no_halo_per_camera(m):
    """Only the ray field R is padded: with every other field of [cameras][voxels] unpadded, one layer of
    512 x 512 voxels and 32 cameras take 0.37 GB (R: 5 x 516^2 x 32 x 4 B; 0.65 GB with two more padded)."""
    torch.cuda.synchronize()
    sc = _scene((512, 512, 1), 32, 3, px=(4, 4))
    m.Grid.from_scene(sc).close()
    before = torch.cuda.mem_get_info()[0]
    grid = m.Grid.from_scene(sc)
    used = before - torch.cuda.mem_get_info()[0]
    grid.close()
    assert used < 0.5e9, used


def test_line_adjoint_on_both_sides_of_its_rule(m):
    """The fixed-field gradient on grids of more and of fewer voxels than the chip has threads at once
    (blocks in turn over the cameras, or camera after camera), against the FP64 oracle at the
    repository's 1e-3."""
    threads = 2048 * torch.cuda.get_device_properties(0).multi_processor_count
    for shape, more in (((32, 32, 38), False), ((threads // 4096 + 1, 64, 64), True)):
        assert (np.prod(shape) > threads) == more
        sc = _scene(shape, 2, 3, px=(5, 4))
        rng = np.random.default_rng(5)
        L = rng.uniform(0.5, 2.0, (2, sc.nvox)) * sc.beta
        meas = rng.uniform(0.0, 1e-4, sc.n_pix)
        grid, beta = m.Grid.from_scene(sc), dev(sc.beta, np.float32)
        out = grid.surrogate_grad(beta, dev(L, np.float64).view(2, -1), beta, m.make_params(synth.Params()), dev(meas, np.float64))
        eg = rel_l2(out["grad"].cpu().numpy(), oracle.surrogate_grad(sc, L, sc.beta, meas)["grad"])
        record(f"line_adjoint{shape}", grad=eg)
        assert eg < 1e-3, (shape, eg)


@pytest.mark.parametrize("px", [(32, 32), (31, 33), (1024, 1)])
def test_back_projection_on_both_sides_of_its_rule(m, px):
    """The fixed-field gradient with a pixel's rays in one thread (1024 pixels a camera and more) and in
    threads of their own, against the FP64 oracle at the repository's 1e-3; the ray segments are counted
    alike."""
    sc = _scene((9, 11, 7), 2, 3, px=px)
    rng = np.random.default_rng(5)
    L = rng.uniform(0.5, 2.0, (2, sc.nvox)) * sc.beta
    meas = rng.uniform(0.0, 1e-4, sc.n_pix)
    grid, beta = m.Grid.from_scene(sc), dev(sc.beta, np.float32)
    out = grid.surrogate_grad(beta, dev(L, np.float64).view(2, -1), beta, m.make_params(synth.Params()), dev(meas, np.float64))
    st = grid.stats()
    assert st["backproj_segments"] == st["pixel_segments"] > 0
    eg = rel_l2(out["grad"].cpu().numpy(), oracle.surrogate_grad(sc, L, sc.beta, meas)["grad"])
    record(f"back_projection{px}", grad=eg)
    assert eg < 1e-3, eg


@pytest.mark.parametrize("shape,paths", [((5, 7, 9), 64), ((64, 65, 66), 400)])
def test_backward_paths_end_in_fields_with_unusable_voxels(m, shape, paths):
    """A NaN or an infinite extinction in the field stops or blinds paths and costs no others: every
    path ends (both kernels), and pixels that no path of theirs brings near stay finite."""
    sc = _scene(shape, 5, 9, px=(33, 33))
    beta = dev(sc.beta, np.float32)
    beta[shape[0] * shape[1] * (shape[2] - 1)] = float("nan")
    beta[-1] = float("inf")
    grid = m.Grid.from_scene(sc)
    p = synth.Params(albedo=0.95, g=0.7, sun_zenith=0.5, sun_azimuth=0.4, seed=21)
    out = grid.render_bmc(beta, m.make_params(p), paths)
    st = grid.stats()
    assert st["lost"] == 0 and st["bmc_paths"] == paths * sc.n_pix and st["bmc_events"] > 0
    assert torch.isfinite(out["images"]).any()
