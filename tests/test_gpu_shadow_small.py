"""Frames with shadow rays on both sides of the line between the one-kernel form
and the rounds (few primitives over the cube of the lights, few samples),
against the one-kernel form, which counting renders use."""
import numpy as np
import pytest

import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,S,lights,res,spp,k", [
    (6144, 8, 1, 40, 2, 1),     # 49,152 segments: the last left to the one kernel
    (6145, 8, 1, 40, 2, 1),
    (768, 8, 2, 40, 2, 2),
    (769, 8, 2, 40, 2, 2),
    (64, 8, 1, 362, 8, 4),      # 1,048,352 samples, and above
    (64, 8, 1, 363, 8, 4),
    (1, 1, 1, 16, 1, 1),
    (64, 3, 16, 24, 3, 8),
])
def test_both_forms(n, S, lights, res, spp, k):
    from paper_2405_10565_gb300.build import build
    build()
    w = scenegen.clustered(n=n, S=S, res=res, spp=spp, n_clusters=max(1, n // 20))
    L = scenegen.point_lights(lights, np.zeros(3), seed=3)
    ctx = hr.hr_create(0)
    try:
        a = hr.hr_asset_create(ctx, w.scene.verts, w.scene.mat, w.scene.shape)
        hr.hr_build_bvh(ctx, a, None)
        img = [np.zeros((res, res, 3), np.float32) for _ in range(2)]
        for i, flags in enumerate((hr.HR_FLAG_SHADOWS, hr.HR_FLAG_SHADOWS | hr.HR_FLAG_COUNT)):
            d = hr.render_desc(w.camera.pack(), L, spp, k, 7, 0, flags)
            st = hr.hr_render(ctx, a, d, img[i], stats=True)
            assert st.stack_overflows == 0
        assert n == 1 or img[1].max() > 0
        # the same operations in the same order; the compiler may contract them differently
        assert np.allclose(img[0], img[1], rtol=1e-5, atol=1e-7), np.abs(img[0] - img[1]).max()
    finally:
        hr.hr_destroy(ctx)
