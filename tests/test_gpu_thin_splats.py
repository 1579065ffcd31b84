"""Precision of the compositing backward on thin ellipses, where A dx and B dy nearly cancel."""
import numpy as np
import pytest
import torch

from paper_2501_12369_gb300 import darb, synth

from gpu_helpers import gpu_forward, to_np

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

U = 2.0 ** -24  # half a unit in the last place of 1 in FP32


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2501_12369_gb300 import build
    build.build()


def _thin_splat(length, aspect, tilt):
    """One splat whose Gaussian has the standard deviation length / 6 pixels along an axis tilted by `tilt`."""
    s = synth.uniform_cube_scene(1, seed=3)
    s.means[:] = [[0.013, -0.021, 0.0]]
    s.scales[:] = np.array([[1.0, 1.0 / aspect, 1.0 / aspect]]) * length / 6 * 6.0 / 500.0
    s.quats[:] = [[np.cos(tilt / 2), 0.0, 0.0, np.sin(tilt / 2)]]
    s.opacities[:] = 0.9
    return s, synth.pinhole((0.0, 0.0, 6.0), 640, 500, 500.0, bg=(0.2, 0.1, 0.4))


def centre_gradient(proj, cam, dl):
    """d loss / d centre of the only record, of upstream gradients dl [3, H, W]: every pair's dx, dy and q by the
    FP32 sequence that defines them, the rest in 64 bits.  With it the standard deviation that independent
    roundings give it.  Per axis, in units of U:
      1.6 times the root of the sum of squares of 2 o s (|A dx| + |B dy|) over the pairs: two roundings
        (sqrt(2 / 3) U) of terms that cancel, the same for a column of up to four pairs (twice);
      0.15 sqrt(number of 8 x 8 tiles reached) times the sum of the 2 o |s (A dx + B dy)| that are left: additions
        in memory (U / sqrt(3) each) to partial sums of at most half, on average a quarter, of it;
      5 times the result and the root of the sum of squares of what is left: the error of s (the profile, T,
        g . S: at most 16 U), common to all pairs or independent."""
    f = np.float32
    (x, y), (A, B, C, o), c = to_np(proj.mean2d)[0], to_np(proj.conic_o)[0], to_np(proj.rgb)[0].astype(np.float64)
    py, px = np.mgrid[0:cam.height, 0:cam.width].astype(f)
    dx, dy = f(x) - (px + f(0.5)), f(y) - (py + f(0.5))

    def fma(a, b, d):  # the product of two FP32 numbers is exact in 64 bits
        return (a.astype(np.float64) * b.astype(np.float64) + d.astype(np.float64)).astype(f)
    q = fma(dx, fma(np.full_like(dx, A), dx, f(2 * B) * dy), f(C) * dy * dy)
    use = (q >= 0) & (q <= 9)
    q, dx, dy = (np.where(use, v, 0).astype(np.float64) for v in (q, dx, dy))
    A, B, C, o = (float(v) for v in (A, B, C, o))
    F = np.exp(-0.5 * q)
    bg = np.array([float(f(b)) for b in cam.bg])
    s = np.where(use, np.tensordot(c - bg, dl.astype(np.float64), 1) * -0.5 * F, 0.0)
    tiles = np.unique((py[use] // 8) * 10000 + px[use] // 8).size
    out = []
    for a, b in ((A, B), (B, C)):
        left = 2 * o * s * (a * dx + b * dy)
        cancels = 2 * o * s * (np.abs(a * dx) + np.abs(b * dy))
        rss = np.sqrt((cancels ** 2).sum()), np.sqrt((left ** 2).sum())
        out.append((left.sum(), U * (1.6 * rss[0] + 0.15 * np.sqrt(tiles) * np.abs(left).sum() + 5 * (abs(left.sum()) + rss[1]))))
    return out


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("length,aspect,tilt", [(400, 10, 0.6), (400, 40, 0.9), (560, 100, 0.5), (560, 200, 0.785), (560, 1000, 2.2)])
def test_centre_gradient_of_thin_splats(length, aspect, tilt, tile):
    """Eight one-signed upstream gradients, two axes: the root mean square of the sixteen errors, in standard
    deviations, is below 2 (above it one time in 10^7)."""
    scene, cam = _thin_splat(length, aspect, tilt)
    r, sd, proj, bins, img = gpu_forward(scene, cam, "gaussian", tile)
    errors = []
    for seed in range(8):
        dl = np.random.default_rng(seed).uniform(0.5, 1.5, (3, cam.height, cam.width)).astype(np.float32)
        got = to_np(darb.darb_render_bwd(proj, 1, bins, cam, r.kparams, tile, img, torch.from_numpy(dl).cuda()))[0]
        errors += [(got[k] - ref) / sigma for k, (ref, sigma) in enumerate(centre_gradient(proj, cam, dl))]
    assert np.sqrt(np.mean(np.square(errors))) <= 2.0, errors


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("length,aspect,tilt", [(900, 2, 0.6), (2400, 3, 0.9)])
def test_conic_gradients_do_not_depend_on_the_order_of_the_tiles(length, aspect, tilt, tile):
    """A splat over most of the image and one-signed upstream gradients: the tiles' sums of s dx^2 and s dy^2 all
    have one sign and that of s dx dy is at most their geometric mean.  With the rounding of every addition kept, a
    result is off by its own last rounding, so that two agree to 2 U; what the additions of up to 5000 lost
    parts lose themselves is some 5000 U^2, below U / 1000."""
    scene, cam = _thin_splat(length, aspect, tilt)
    r, sd, proj, bins, img = gpu_forward(scene, cam, "gaussian", tile)
    dl = np.random.default_rng(3).uniform(0.5, 1.5, (3, cam.height, cam.width)).astype(np.float32)
    dl = torch.from_numpy(dl).cuda()
    got = np.stack([to_np(darb.darb_render_bwd(proj, 1, bins, cam, r.kparams, tile, img, dl))[0] for _ in range(24)])
    assert (got[:, 9:] == 0).all()
    a, b, c = (got[:, k].astype(np.float64) for k in (2, 3, 4))
    for v, size in ((a, np.abs(a).max()), (c, np.abs(c).max())):
        assert np.ptp(v) <= 2.01 * U * size
    assert np.ptp(b) <= 2 * U * np.abs(b).max() + 0.01 * U * np.sqrt(np.abs(a).max() * np.abs(c).max())
