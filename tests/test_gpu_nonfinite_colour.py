"""A splat whose colour is not finite, or so large that products with it overflow, reaches only the pixels that
blend it, and in the backward only the splats that those pixels blend."""
import numpy as np
import pytest
import torch

from paper_2501_12369_gb300 import darb, synth

from gpu_helpers import gpu_forward, to_np

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2501_12369_gb300 import build
    build.build()


@pytest.mark.parametrize("kernel", ["half_cosine", "raised_cosine"])
@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("bad", [np.inf, np.nan, 3e38])
def test_colour_that_is_not_finite_stays_where_it_is_blended(bad, tile, kernel):
    s = synth.cluster_scene(4000, seed=8, sh_degree=0)
    s.opacities[:] = np.minimum(1.0, s.opacities * 2.0)  # most pixels stop well before their list's end
    cam = synth.fibonacci_cameras(16, 6.0, 150, 97, 120.0)[2]
    r, sd, proj, bins, img = gpu_forward(s, cam, kernel, tile)
    dl = synth.random_image_grad(97, 150, seed=4)

    def render():
        return darb.darb_render_fwd(proj, bins, cam, r.kparams, tile)

    def backward(img, dl):
        return to_np(darb.darb_render_bwd(proj, s.n, bins, cam, r.kparams, tile, img,
                                          torch.from_numpy(np.ascontiguousarray(dl, np.float32)).cuda()))
    clean, clean_g, colours = to_np(img.image), backward(img, dl), proj.rgb.clone()
    reach = to_np(proj.tiles_touched).astype(np.int64)
    behind = stopped_before = 0
    for i in np.argsort(-reach)[[0, 3, 20, 100, 400]]:
        proj.rgb.zero_()
        proj.rgb[i] = 1.0
        blends = to_np(render().image)[0] > 0  # the background is black
        proj.rgb.copy_(colours)
        proj.rgb[i, 1] = bad
        out = render()
        image = to_np(out.image)
        assert np.array_equal(image[:, ~blends], clean[:, ~blends])
        assert np.array_equal(image[[0, 2]], clean[[0, 2]])
        assert not np.isfinite(bad) or np.isfinite(image).all()
        assert np.isfinite(bad) or not np.isfinite(image[1][blends]).any()
        target = torch.from_numpy(synth.random_target(97, 150, seed=9)).cuda()
        l1 = darb.darb_render_fwd_l1(proj, bins, cam, r.kparams, tile, target)[0]
        assert np.array_equal(to_np(l1.image), image, equal_nan=True)
        touched = (backward(out, np.broadcast_to(blends, (3, 97, 150)))[:, 6:9] != 0).any(axis=1)
        got = backward(out, dl)
        assert np.isfinite(got[~touched]).all()
        np.testing.assert_allclose(got[~touched], clean_g[~touched], rtol=1e-4, atol=1e-5 * np.abs(clean_g).max())
        behind += int(blends.sum())
        stopped_before += int((~blends).sum())
        proj.rgb.copy_(colours)
    assert behind > 0 and stopped_before > 0
