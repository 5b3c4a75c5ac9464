"""A frame's image does not depend on which kernel finishes a ray, nor on the order
of its tests: frames repeat bit for bit, also where the room for the rays put
aside runs out (which of them find some is a matter of timing), and equal
counting frames, which put none aside."""
import numpy as np
import pytest

import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,S,clusters,res,spp,k,setting", [
    (4000, 16, 400, 96, 4, 8, "half"),    # the records of K = 8 outgrow the room of so small a frame
    (20000, 32, 1000, 160, 4, 8, "half"),
    (60000, 32, 3000, 128, 8, 8, "eth"),
    (20000, 64, 5000, 200, 8, 8, "eth"),
    (4000, 16, 400, 48, 3, 2, "half"),
    (4000, 16, 400, 33, 32, 1, "eth"),
])
def test_frames_repeat_whichever_rays_are_put_aside(n, S, clusters, res, spp, k, setting):
    from paper_2405_10565_gb300.build import build
    build()
    w = scenegen.clustered(n=n, S=S, res=res, spp=spp, lod_setting=setting, n_clusters=clusters)
    ctx = hr.hr_create(0)
    try:
        a = hr.hr_asset_create(ctx, w.scene.verts, w.scene.mat, w.scene.shape)
        hr.hr_build_clusters(ctx, a, w.n_clusters)
        C, L, _ = hr.hr_hierarchy_info(ctx, a)
        hr.hr_build_bvh(ctx, a, scenegen.lod_preset(setting, C, L))
        frames, used = [], []
        for flags in [hr.HR_FLAG_COUNT] + [0] * 10 + [hr.HR_FLAG_FIXED_TILE_ORDER] * 2:
            frames.append(np.zeros((res, res, 3), np.float32))
            hr.hr_render(ctx, a, hr.render_desc(w.camera.pack(), w.lights, spp, k, 5, 0, flags), frames[-1])
            used.append(hr.hr_bytes_in_use(ctx))
    finally:
        hr.hr_destroy(ctx)
    assert used[1] > used[0] + 65536  # the first that may put rays aside took room for them
    assert frames[0].max() > 0
    assert all(np.array_equal(f, frames[0]) for f in frames), [int((f != frames[0]).sum()) for f in frames]
