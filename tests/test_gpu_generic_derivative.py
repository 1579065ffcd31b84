"""dF/dq of single pixels against 64 bits."""
import numpy as np
import pytest
import torch

from paper_2501_12369_gb300 import darb, synth

from gpu_helpers import to_np

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2501_12369_gb300 import build
    build.build()


def _one_pixel():
    """One record and one pixel that its gradients come from: projected records, lists, images, upstream
    gradient (1 in red) and camera."""
    cam = synth.pinhole((0.0, 0.0, 4.0), 8, 8, 8.0)
    proj = darb.Projected.empty(1, "cuda")
    bins = darb.Binning.empty(16, 1, "cuda")
    bins.values.zero_()
    bins.ranges[:] = torch.tensor([[0, 1]], dtype=torch.int32)
    img = darb.ImageOut.empty(8, 8, "cuda")
    img.last.zero_()
    img.last[0, 0] = 1
    img.t_final.fill_(1.0)
    dl = torch.zeros(3, 8, 8, device="cuda")
    dl[0, 0, 0] = 1.0
    for name in ("radius", "tiles_touched"):
        getattr(proj, name).fill_(1)
    proj.rgb[:] = torch.tensor([[1.0, 0.0, 0.0]])
    proj.conic_o[:] = torch.tensor([[1.0, 0.0, 1.0, 0.5]])
    return cam, proj, bins, img, dl


def test_derivative_of_a_linear_profile_in_the_distance_is_exact():
    """F = 1 - sqrt(q) / xi at one pixel with dx = m, dy = 0 and the unit conic: q = m^2, and with 1 / xi = m / 2^k
    u = m^2 / 2^k, so that u / q = 2^-k and dF/dq = -2^-(k + 1) need no rounding.  The gradients of that pixel
    are then m dF T and (with alpha = F / 2 = 1 - T before the replay) alpha T in red, each rounded once, T
    the replayed transmittance, 1 but for its own rounding, which is the same in both."""
    f = np.float32
    cam, proj, bins, img, dl = _one_pixel()
    for m in range(3, 259, 2):
        k = int(np.ceil(2 * np.log2(m))) + 2
        inv_xi = f(m) * f(2.0) ** -k
        near = f(1.0) / inv_xi
        xi = [x for x in (near, np.nextafter(near, f(0)), np.nextafter(near, f(1e9))) if f(1.0) / x == inv_xi]
        if not xi:  # no FP32 number has this inverse: 26 of the 128
            continue
        kp = darb.darb_kernel_generic("parabola", float(xi[0]), 1.0, 1, 1.0)
        kp.q_max = 1e5
        alpha = f(0.5) * (f(1.0) - f(m * m) * f(2.0) ** -k)
        img.t_final[0, 0] = float(f(1.0) - alpha)
        proj.mean2d[:] = torch.tensor([[0.5 + m, 0.5]])
        g = to_np(darb.darb_render_bwd(proj, 1, bins, cam, kp, 8, img, dl))[0]
        near1 = [f(1.0) + f(j) * f(2.0) ** -24 for j in (-4, -3, -2, -1, 0, 2, 4)]
        replayed = [t for t in near1 if alpha * t == g[6]]
        assert replayed, (m, g[6], alpha)
        assert g[0] in [-f(m) * t * f(2.0) ** -(k + 1) for t in replayed], (m, g[0])


def test_derivative_of_the_raised_cosine():
    """q from 1e-4 to 1, with dx = 8 and dy = 0.  The gradients w.r.t. centre and opacity are 8 dF g and F g, g the
    same in both: their quotient is 8 dF / F.  F's cosine is off by 2^-21.2, of F >= 0.65 by 7e-7 / 1.3; nine
    roundings of the series, of terms that decrease, and eight of products are 1e-6 at most."""
    f = np.float32
    cam, proj, bins, img, dl = _one_pixel()
    kp = darb.darb_kernel_defaults("raised_cosine")
    proj.mean2d[:] = torch.tensor([[8.5, 0.5]])
    k = np.pi / 2.5
    for q in np.geomspace(1e-4, 1.0, 97):
        A = f(q / 64)  # dx^2 is a power of two: q is exact
        q = 64.0 * float(A)
        proj.conic_o[:] = torch.tensor([[float(A), 0.0, 1.0, 0.5]])
        F, dF = 0.5 + 0.5 * np.cos(k * np.sqrt(q)), -k / 4 * np.sin(k * np.sqrt(q)) / np.sqrt(q)
        img.t_final[0, 0] = 1 - 0.5 * F
        g = to_np(darb.darb_render_bwd(proj, 1, bins, cam, kp, 8, img, dl))[0].astype(np.float64)
        want = 8 * float(A) * dF / F
        assert abs(g[0] / g[5] - want) <= 1.6e-6 * abs(want), (q, g[0] / g[5], want)


def test_derivative_of_the_raised_cosine_past_its_main_lobe():
    """A caller's q_max of 60: __sinf is off by 2^-20 at x <= 10, of |sin x| >= 0.1, and F >= 0.1 by 2^-20: 2e-5."""
    cam, proj, bins, img, dl = _one_pixel()
    kp = darb.darb_kernel_defaults("raised_cosine")
    kp.q_max = 60.0
    proj.mean2d[:] = torch.tensor([[8.5, 0.5]])
    k, seen = np.pi / 2.5, 0
    for q in np.linspace(5.0, 60.0, 111):
        A = np.float32(q / 64)
        q = 64.0 * float(A)
        proj.conic_o[:] = torch.tensor([[float(A), 0.0, 1.0, 0.5]])
        F, dF = 0.5 + 0.5 * np.cos(k * np.sqrt(q)), -k / 4 * np.sin(k * np.sqrt(q)) / np.sqrt(q)
        if F < 0.1 or abs(np.sin(k * np.sqrt(q))) < 0.1:
            continue
        seen += 1
        img.t_final[0, 0] = 1 - 0.5 * F
        g = to_np(darb.darb_render_bwd(proj, 1, bins, cam, kp, 8, img, dl))[0].astype(np.float64)
        want = 8 * float(A) * dF / F
        assert abs(g[0] / g[5] - want) <= 2e-5 * abs(want), (q, g[0] / g[5], want)
    assert seen > 40
