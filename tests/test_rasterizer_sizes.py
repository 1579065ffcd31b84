"""The buffers a Rasterizer hands to the sort, for a camera or a tile that is changed between calls (on the CPU:
the launches are replaced by a function that looks at the buffers)."""
import pytest

from paper_2501_12369_gb300 import build, darb, synth


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("strategy", [darb.DARB_SORT_DEPTH_THEN_TILE, darb.DARB_SORT_KEYS64])
@pytest.mark.parametrize("owned", [False, True])
def test_lists_and_workspace_fit_the_present_camera_and_tile(monkeypatch, strategy, owned):
    s = synth.uniform_cube_scene(100)
    big, small = (synth.pinhole((0.0, 0.0, 4.0), w, h, 500.0) for w, h in ((1920, 1080), (333, 207)))
    seen = []

    def sort(proj, n, tile, cam, workspace, capacity, out, **kw):
        tx, ty = darb.darb_tile_grid(cam, tile)
        seen.append((tile, cam.width, out.ranges.shape[0] - tx * ty, out.values.shape[0] - capacity,
                     workspace.numel() >= darb.darb_bin_sort_workspace_size(n, tile, cam, capacity, kw["strategy"])))
        return out
    monkeypatch.setattr(darb, "darb_preprocess", lambda *a: None)
    monkeypatch.setattr(darb, "darb_bin_sort", sort)
    monkeypatch.setattr(darb, "darb_render_fwd", lambda *a: None)
    r = darb.Rasterizer(big, "half_cosine", 32, capacity=1 << 16, device="cpu", strategy=strategy)
    want = []
    for tile, cam in ((32, big), (8, big), (16, big), (16, small), (8, small), (8, big)):
        r.tile, r.cam = tile, cam
        r.forward(s, owned=owned)
        want.append((tile, cam.width, 0, 0, True))
    assert seen == want
