"""Frames with shadow rays by separate hit, light-path and shading kernels
against the one-kernel form (which counting renders use): one round, several
rounds with tiles left over, more samples than lanes of a pixel, K of every
kernel width, and a context whose memory budget has no room for the rounds."""
import numpy as np
import pytest

import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("res,spp,k,lights,setting,budget", [
    (37, 3, 1, 1, "half", 0),
    (64, 1, 2, 3, "strands", 0),
    (48, 8, 3, 2, "half", 0),
    (16, 40, 4, 2, "half", 0),       # a lane takes two samples: the one-kernel form
    (640, 8, 8, 16, "eth", 0),       # over 2^20 hits a round: three rounds and a rest
    (64, 4, 4, 4, "half", 1),        # no memory for the rounds
])
def test_rounds_equal_the_one_kernel_form(res, spp, k, lights, setting, budget):
    from paper_2405_10565_gb300.build import build
    build()
    w = scenegen.clustered(n=1500, S=8, res=res, spp=spp, lod_setting=setting, n_clusters=40)
    L = scenegen.point_lights(lights, np.zeros(3), seed=3)
    ctx = hr.hr_create(0)
    try:
        def scene(c):
            a = hr.hr_asset_create(c, w.scene.verts, w.scene.mat, w.scene.shape)
            hr.hr_build_clusters(c, a, w.n_clusters)
            C, n_levels, _ = hr.hr_hierarchy_info(c, a)
            hr.hr_build_bvh(c, a, scenegen.lod_preset(setting, C, n_levels))
            return a
        a = scene(ctx)
        img = [np.zeros((res, res, 3), np.float32) for _ in range(3)]
        for i, flags in enumerate((hr.HR_FLAG_SHADOWS, hr.HR_FLAG_SHADOWS | hr.HR_FLAG_COUNT)):
            d = hr.render_desc(w.camera.pack(), L, spp, k, 7, 0, flags)
            st = hr.hr_render(ctx, a, d, img[i], stats=True)
            assert st.stack_overflows == 0
        assert img[1].max() > 0
        if setting == "eth":
            assert st.shaded_hits > 4 << 20
        # the same operations in the same order; the compiler may contract them differently
        assert np.allclose(img[0], img[1], rtol=1e-5, atol=1e-7), np.abs(img[0] - img[1]).max()
        if budget:
            probe = hr.hr_create(0)
            b = scene(probe)
            hr.hr_render(probe, b, hr.render_desc(w.camera.pack(), L, spp, k, 7, 0, 0), img[2])
            tight = hr.hr_bytes_in_use(probe)
            hr.hr_destroy(probe)
            tctx = hr.hr_create(0, tight + 4096)
            b = scene(tctx)
            d = hr.render_desc(w.camera.pack(), L, spp, k, 7, 0, hr.HR_FLAG_SHADOWS)
            hr.hr_render(tctx, b, d, img[2])
            assert hr.hr_bytes_in_use(tctx) <= tight + 4096
            hr.hr_destroy(tctx)
            assert np.allclose(img[2], img[0], rtol=1e-5, atol=1e-7)
    finally:
        hr.hr_destroy(ctx)
