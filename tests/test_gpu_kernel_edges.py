"""Edges of the kernels' tilings and of the rules that choose between their variants."""
import numpy as np
import pytest
import torch

import oracle
from paper_2501_12369_gb300 import darb, synth

from gpu_helpers import ambiguity_masked_grad, check_lists, check_preprocess, check_render, gpu_forward, grad_close, to_np
from test_gpu_density import CFG, RAW, STATE_OF, _case, _device, _t

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2501_12369_gb300 import build
    build.build()
    oracle.build()


def _off_by_one(t):
    """The same values 4 bytes past a 16-byte boundary."""
    flat = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    v = flat[1:].view(t.shape)
    v.copy_(t)
    assert v.data_ptr() % 16 == 4
    return v


@pytest.mark.parametrize("n", [1, 511, 512, 513, 2048, 2049, 4100])
@pytest.mark.parametrize("deg", [0, 2, 3])
def test_densify_at_block_edges_with_unaligned_moments(n, deg):
    """Row counts around a scatter CTA's 512 and a counted block's 2048 splats, SH rows that are and are
    not multiples of 16 bytes, and moments off the 16-byte boundary (the parameters must be on it)."""
    raw, act, state, accum, count, radius, normals = _case(n, deg, seed=20 + deg)
    ref_raw, ref_act, ref_state, n_ref = oracle.densify(raw, act, state, accum, count, radius, normals, CFG)
    p, st = _device(raw, act, state, deg)
    po, so = _device(raw, act, state, deg, rows=2 * n)
    for s in (st, so):
        for f, t in vars(s).items():
            setattr(s, f, _off_by_one(t))
    n_out = darb.darb_densify(p, st, _t(accum), _t(count), _t(radius), _t(normals), darb.darb_densify_cfg(**CFG), po, so)
    torch.cuda.synchronize()
    rows, _, children = (int(x) for x in to_np(n_out))
    assert rows == n_ref
    for k in RAW:
        got, exact = to_np(getattr(po, k)), children if k == "means" else rows
        np.testing.assert_array_equal(got[:exact], ref_raw[k][:exact], err_msg=k)
        np.testing.assert_allclose(got[:rows], ref_raw[k], rtol=0, atol=2e-6)
        assert np.isnan(got[rows:]).all(), "rows past the output were written"
        for m in ("m", "v"):
            mom = to_np(getattr(so, f"{m}_{STATE_OF[k]}"))
            np.testing.assert_array_equal(mom[:rows], ref_state[f"{m}_{k}"])
            assert np.isnan(mom[rows:]).all()


@pytest.mark.parametrize("kernel", ["gaussian", "mod_sinc", "raised_cosine"])
@pytest.mark.parametrize("tile,width,height", [(32, 992, 511), (32, 1000, 513), (16, 1, 1), (16, 17, 16), (8, 63, 9)])
def test_compositing_backward_on_either_side_of_its_block_rule(kernel, tile, width, height):
    """992 x 511 has 3968 blocks of 16 x 8 pixels per 32-pixel tiles (four pixels a lane), 1000 x 513 has 4352;
    fewer than 3952 take two pixels a lane.  Very small images leave most of a block outside."""
    s = synth.cluster_scene(1500, seed=31, sh_degree=0)
    cam = synth.pinhole((0.5, 0.4, 6.0), width, height, 0.8 * max(width, 24), bg=(0.2, 0.1, 0.4))
    r, sd, proj, bins, img = gpu_forward(s, cam, kernel, tile)
    ref = oracle.forward(s, cam, kernel, tile=tile)
    check_render(img, bins, ref, cam, tile)
    dl = ambiguity_masked_grad(synth.random_image_grad(height, width, seed=4), ref["amb"])
    _, g2, _ = oracle.gradients(s, cam, dl, kernel, tile=tile)
    got = darb.darb_render_bwd(proj, s.n, bins, cam, r.kparams, tile, img, _t(dl.astype(np.float32)))
    torch.cuda.synchronize()
    for u in range(9):
        grad_close(f"grad2d[{u}]", to_np(got)[:, u], np.asarray(g2)[:, u])


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("n", [96, 97, 128, 129, 300])
def test_compositing_backward_at_the_edges_of_its_windows(n, tile):
    """Faint splats that all cover the image, so that every pixel's run is as long as the list: windows are
    of 96 records (32-pixel tiles) and 128."""
    s = synth.uniform_cube_scene(n, seed=5, half=0.3, log_scale=(-0.5, 0.5))
    s.opacities[:] = np.linspace(0.008, 0.016, n, dtype=np.float32)
    cam = synth.pinhole((0.5, 0.4, 6.0), 40, 33, 60.0, bg=(0.2, 0.1, 0.4))
    r, sd, proj, bins, img = gpu_forward(s, cam, "gaussian", tile)
    ref = oracle.forward(s, cam, "gaussian", tile=tile)
    check_render(img, bins, ref, cam, tile)
    assert int(img.n_contrib.max()) > 0.9 * n
    dl = ambiguity_masked_grad(synth.random_image_grad(33, 40, seed=4), ref["amb"])
    _, g2, _ = oracle.gradients(s, cam, dl, "gaussian", tile=tile)
    got = darb.darb_render_bwd(proj, s.n, bins, cam, r.kparams, tile, img, _t(dl.astype(np.float32)))
    torch.cuda.synchronize()
    for u in range(9):
        grad_close(f"grad2d[{u}]", to_np(got)[:, u], np.asarray(g2)[:, u])


@pytest.mark.parametrize("kernel", ["gaussian", "mod_sinc"])
@pytest.mark.parametrize("width,height", [(960, 544), (1280, 720), (1312, 720)])
def test_compositing_backward_block_rule_of_16_pixel_tiles(kernel, width, height):
    """Fewer than 7296 blocks of 16 x 8 pixels take two pixels a lane: 4080, 7200 and 7380 blocks."""
    test_compositing_backward_on_either_side_of_its_block_rule(kernel, 16, width, height)


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_gradient_that_is_not_finite_stays_with_the_splats_its_pixel_blended(bad):
    s = synth.cluster_scene(4000, seed=8, sh_degree=0)
    cam = synth.fibonacci_cameras(16, 6.0, 150, 97, 120.0)[2]
    r, sd, proj, bins, img = gpu_forward(s, cam, "half_cosine", 16)
    dl = synth.random_image_grad(97, 150, seed=4)
    clean = to_np(darb.darb_render_bwd(proj, s.n, bins, cam, r.kparams, 16, img, _t(dl)))
    y, x = 50, 75
    one = np.zeros_like(dl)
    one[:, y, x] = 1.0
    touched = (to_np(darb.darb_render_bwd(proj, s.n, bins, cam, r.kparams, 16, img, _t(one)))[:, 6:9] != 0).any(axis=1)
    dl[1, y, x] = bad
    got = to_np(darb.darb_render_bwd(proj, s.n, bins, cam, r.kparams, 16, img, _t(dl)))
    assert 0 < touched.sum() < s.n
    assert not np.isfinite(got[touched]).all(axis=1).any()
    assert np.isfinite(got[~touched]).all()
    np.testing.assert_allclose(got[~touched], clean[~touched], rtol=1e-4, atol=1e-5 * np.abs(clean).max())


@pytest.mark.parametrize("kernel", oracle.KERNEL_NAMES)
def test_conic_that_rounds_to_indefinite_adds_nothing_outside_its_support(kernel):
    """A record whose conic is not positive definite in FP32 has q far below 0 (where the Gaussian overflows)
    and far above its limit (where the sinc's series does): such pairs carry weight 0 and every gradient
    stays finite and as it is without the record."""
    s = synth.cluster_scene(500, seed=3, sh_degree=0)
    cam = synth.pinhole((0.0, 0.0, 6.0), 64, 48, 60.0)
    r, sd, proj, bins, img = gpu_forward(s, cam, kernel, 16)
    lists, ranges = to_np(bins.values), to_np(bins.ranges)
    first = np.unique([lists[a] for a, b in ranges if b > a])  # the nearest record of every tile
    proj.conic_o[torch.from_numpy(first.astype(np.int64)).cuda()] = torch.tensor([1e6, 3e6, 1e6, 0.5], device="cuda")
    proj.mean2d[torch.from_numpy(first.astype(np.int64)).cuda()] += 1000.25
    img = darb.darb_render_fwd(proj, bins, cam, r.kparams, 16)
    assert torch.isfinite(img.image).all()
    g = to_np(darb.darb_render_bwd(proj, s.n, bins, cam, r.kparams, 16, img, _t(synth.random_image_grad(48, 64, seed=4))))
    assert np.isfinite(g).all() and (g[first] == 0).all() and np.abs(g).max() > 0


@pytest.mark.parametrize("n", [1, 31, 1025, 2048, 2049, 16384, 16385, 32768, 32769])
def test_depth_order_of_small_scenes_at_the_edges_of_its_cluster(n):
    """2048 positions a CTA and up to 8 CTAs to 16384 splats, 4096 to 32768, the passes of any size beyond; with equal depths (which keep splat order) and culled splats."""
    s = synth.cluster_scene(n, seed=n, sh_degree=0)
    s.means[::7] = s.means[0]
    s.means[3::11, :] *= np.float32(40.0)  # outside the frame or behind the camera
    cam = synth.fibonacci_cameras(16, 6.0, 205, 121, 160.0)[5]
    r, sd, proj, bins, img = gpu_forward(s, cam, "half_cosine", 16)
    ref = oracle.project(s, cam, oracle.kernel_params("half_cosine"), 16, True)
    lists = oracle.build_lists(ref, cam, 16)
    check_lists(bins, lists)
    if lists["M"] > 1:  # one instance too many, found on the device
        cap = lists["M"] - 1
        ws = torch.empty(darb.darb_bin_sort_workspace_size(n, 16, cam, cap), dtype=torch.uint8, device="cuda")
        b = darb.darb_bin_sort(proj, n, 16, cam, ws, cap, sync=False)
        torch.cuda.synchronize()
        assert int(to_np(b.status)[0]) == 3 and int(to_np(b.num_instances)[0]) == lists["M"]
        assert (to_np(b.ranges) == 0).all()


@pytest.mark.parametrize("width,height", [(5, 3), (31, 33), (32, 32), (33, 65), (1300, 700)])
def test_dssim_at_tile_edges(width, height):
    """Images smaller than a halo, one tile, just over it, and (1300 x 700) more tiles than the backward has CTAs."""
    img, tgt = synth.random_target(height, width, seed=5), synth.random_target(height, width, seed=6)
    img[:, ::2] = tgt[:, ::2]
    dl, loss = darb.darb_l1_dssim_loss(_t(img), _t(tgt), 0.2)
    ref_loss, ref_dl, ref_ssim = oracle.l1_dssim_loss(img, tgt, 0.2)
    torch.cuda.synchronize()
    assert abs(float(loss[0]) - ref_loss) <= 2e-6 and abs(float(loss[1]) - ref_ssim) <= 4e-6
    grad_close("dL", to_np(dl), ref_dl)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 300])
@pytest.mark.parametrize("deg", [0, 1, 2, 3])
def test_preprocess_backward_stores_at_block_edges_and_off_the_boundary(n, deg):
    """Gradients leave a block of 128 splats as contiguous ranges: ragged last blocks, and arrays 4 bytes past
    a 16-byte boundary, give the values of aligned ones."""
    s = synth.uniform_cube_scene(n, seed=deg, sh_degree=deg)
    cam = synth.pinhole((0.0, 0.0, 4.0), 64, 48, 60.0)
    sd = darb.splats_to_device(s)
    kp = darb.darb_kernel_defaults("half_cosine")
    proj = darb.darb_preprocess(sd, cam, kp, 16)
    g2 = _t(np.random.default_rng(n).normal(size=(n, 12)).astype(np.float32))
    a = darb.darb_preprocess_bwd(sd, cam, kp, proj, g2)
    b = darb.SplatGrads.empty_like(sd)
    for f in ("dmeans", "dscales", "dopacities"):
        setattr(b, f, _off_by_one(torch.full_like(getattr(b, f), np.nan)))
    darb.darb_preprocess_bwd(sd, cam, kp, proj, g2, b)
    torch.cuda.synchronize()
    seen = to_np(proj.radius) > 0
    assert seen.any()
    for f in ("dmeans", "dscales", "dquats", "dopacities", "dsh"):
        x, y = to_np(getattr(a, f)), to_np(getattr(b, f))
        np.testing.assert_array_equal(x, y, err_msg=f)
        assert (x[~seen] == 0).all() and np.isfinite(x).all()


@pytest.mark.parametrize("n", [1, 2, 683, 2049])
@pytest.mark.parametrize("deg", [0, 2, 3])
def test_adam_groups_at_block_edges(n, deg):
    """Groups shorter than a float4 and just over a block's 2048 floats (3 x 683 and 2049): every element
    takes exactly one step."""
    from test_gpu_train import _cfg, _check_adam, _clone, _oracle_adam, _to_device, _train_state
    s = synth.uniform_cube_scene(n, seed=deg, sh_degree=deg)
    rng = np.random.default_rng(50 + deg)
    raw, state = _train_state(s, rng, warm=True)
    p, st = _to_device(raw, state, deg)
    p0, _ = _clone(p, st)
    grads = {k: (1e-3 * rng.normal(size=getattr(s, k).shape)).astype(np.float32)
             for k in ("means", "scales", "quats", "opacities", "sh")}
    ref_raw, ref_state = _oracle_adam(p, st, {k: v.astype(np.float64) for k, v in grads.items()}, 5)
    darb.darb_adam_step(p, darb.SplatGrads(*(_t(grads[k]) for k in ("means", "scales", "quats", "opacities", "sh"))), st,
                        _cfg(5))
    torch.cuda.synchronize()
    _check_adam(p0, p, st, ref_raw, ref_state, upd_rtol=1e-5, mom_tol=2e-6)


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("width,height", [(1, 1), (128, 16), (16, 129), (333, 207)])
def test_l1_epilogue_loss_at_cluster_edges(width, height, tile):
    """Fewer CTAs than a cluster of 8, whole clusters and a last one that is not full.  Every thread adds at most
    12 terms, and no term goes through more than 12 + 5 + 8 + 8 additions before those in memory (at
    most 135 clusters): (33 + 135) 2^-24 < 1.1e-5 of the loss, whose terms are all positive."""
    s = synth.uniform_cube_scene(300, seed=6)
    cam = synth.pinhole((0.5, 0.4, 6.0), width, height, 0.8 * max(width, 24), bg=(0.2, 0.1, 0.4))
    r, sd, proj, bins, img = gpu_forward(s, cam, "gaussian", tile)
    target = _t(synth.random_target(height, width, seed=9))
    out, dl, loss = darb.darb_render_fwd_l1(proj, bins, cam, r.kparams, tile, target)
    torch.cuda.synchronize()
    d = to_np(out.image).astype(np.float64) - to_np(target)
    assert abs(float(loss[0]) - np.abs(d).mean()) <= 1.1e-5 * np.abs(d).mean()
    np.testing.assert_array_equal(to_np(out.image), to_np(img.image))
    np.testing.assert_array_equal(to_np(dl), np.sign(d).astype(np.float32) * np.float32(1.0 / (3.0 * width * height)))


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("n", [1, 33, 700])
def test_member_tiles_of_tall_rectangles(n, tile):
    """Splats from a pixel to the whole image: rectangles within a packed word's 8 rows, a few taller ones beside
    them and warps of tall ones, up to 163 rows (more than a warp's lanes)."""
    s = synth.uniform_cube_scene(n, seed=12, half=1.5, log_scale=(-5.0, 0.7))
    s.scales[::32] = 1.0
    cam = synth.pinhole((0.5, 0.4, 6.0), 333, 1300, 600.0, bg=(0.2, 0.1, 0.4))
    r, sd, proj, bins, img = gpu_forward(s, cam, "gaussian", tile)
    ref = oracle.project(s, cam, oracle.kernel_params("gaussian"), tile, True)
    rect = to_np(proj.tile_rect)[0]
    assert rect[3] - rect[1] + 1 > 8
    check_preprocess(proj, ref)
