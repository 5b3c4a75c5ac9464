"""Memory of a frame with shadow rays: 448 MB of hits and light paths at most and
40 bytes a warp tile, whatever the number of lights and the depth of the k-buffer;
the image is that of a counting frame, which needs none of it."""
import numpy as np
import pytest

import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,spp,k,lights", [
    (1920, 1080, 8, 4, 1),
    (1920, 1080, 8, 8, 16),
    (3840, 2160, 1, 2, 2),
    (1921, 33, 32, 8, 3),
    (160, 90, 4, 8, 8),       # the worst case fits
])
def test_bytes_of_a_shadow_frame(W, H, spp, k, lights):
    from paper_2405_10565_gb300.build import build
    build()
    w = scenegen.clustered(n=2500, S=24, res=64, spp=spp, lod_setting="half", n_clusters=200)
    cam = scenegen.frame_camera(*w.scene.aabb(), W, H, perspective=True, fill=0.05 if W > 1000 else 0.6)
    L = scenegen.point_lights(lights, np.zeros(3), seed=3)
    ctx = hr.hr_create(0)
    try:
        a = hr.hr_asset_create(ctx, w.scene.verts, w.scene.mat, w.scene.shape)
        hr.hr_build_clusters(ctx, a, w.n_clusters)
        C, levels, _ = hr.hr_hierarchy_info(ctx, a)
        hr.hr_build_bvh(ctx, a, scenegen.lod_preset("half", C, levels))
        img, used = [], []
        for flags in (hr.HR_FLAG_SHADOWS | hr.HR_FLAG_COUNT, hr.HR_FLAG_SHADOWS):
            img.append(np.zeros((H, W, 3), np.float32))
            hr.hr_render(ctx, a, hr.render_desc(cam.pack(), L, spp, k, 7, 0, flags), img[-1])
            used.append(hr.hr_bytes_in_use(ctx))
        warp_tiles = (W // 4 + 1) * (H // 4 + 1) * (16 // (32 // min(32, 1 << (spp - 1).bit_length())) + 1)
        worst = W * H * spp * k * (20 + 16 * lights)
        assert 0 < used[1] - used[0] <= min(448 << 20, worst) + 40 * warp_tiles + 4096
        assert img[0].max() > 0
        assert np.allclose(img[1], img[0], rtol=1e-5, atol=1e-7)  # as for the rounds
    finally:
        hr.hr_destroy(ctx)
