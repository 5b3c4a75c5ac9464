"""The tile schedule of frames that hand out parts of tiles: a tile with several
heavy parts is one heavy tile."""
import numpy as np
import pytest

import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,spp", [(8, 4, 1), (5, 3, 1), (4, 4, 8), (11, 9, 2), (16, 12, 4)])
def test_heavy_tiles_are_tiles(W, H, spp):
    from paper_2405_10565_gb300.build import build
    build()
    w = scenegen.clustered(n=4000, S=16, res=64, spp=spp, lod_setting="half", n_clusters=400)
    cam = scenegen.frame_camera(*w.scene.aabb(), W, H, perspective=True, fill=1.2)
    ctx = hr.hr_create(0)
    try:
        a = hr.hr_asset_create(ctx, w.scene.verts, w.scene.mat, w.scene.shape)
        hr.hr_build_clusters(ctx, a, w.n_clusters)
        C, L, _ = hr.hr_hierarchy_info(ctx, a)
        hr.hr_build_bvh(ctx, a, scenegen.lod_preset("half", C, L))
        d = hr.render_desc(cam.pack(), w.lights, spp, 4, 7)
        img = [np.zeros((H, W, 3), np.float32) for _ in range(5)]
        heavy = [hr.hr_render(ctx, a, d, i, stats=True).heavy_tiles for i in img]
        px = 32 // min(32, 1 << (spp - 1).bit_length())  # pixels of a warp tile
        tw = 1
        while tw * tw < px:
            tw *= 2
        tiles = -(-W // tw) * -(-H // (px // tw))
        print(W, H, spp, tiles, heavy)
        assert heavy[0] == 0 and max(heavy) > 0
        assert max(heavy) <= tiles
        assert img[0].max() > 0 and all(np.array_equal(i, img[0]) for i in img)
    finally:
        hr.hr_destroy(ctx)
