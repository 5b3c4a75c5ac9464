"""Device memory of a BVH build: a node's FP32 boxes (64 bytes a leaf), its links
and ids (28) and, with the sort's keys and values, scratch with a quarter on top.
A context whose budget held this much for a scene goes on building it."""
import numpy as np
import pytest

import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,S", [(10, 30), (40, 8), (2500, 16), (20000, 32)])
def test_bytes_a_leaf(n, S):
    from paper_2405_10565_gb300.build import build
    build()
    v = scenegen.make_strands(n, S, seed=1)
    ctx = hr.hr_create(0)
    try:
        a = hr.hr_asset_create(ctx, v, scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2)),
                               np.zeros((n, 2), np.float32))
        before = hr.hr_bytes_in_use(ctx)
        hr.hr_build_bvh(ctx, a, None)
        used = hr.hr_bytes_in_use(ctx) - before
        # 92 kept; ids, keys and their temporaries 4 * 4, links of the climb 8, boxes 32; and small ones
        assert used <= n * S * (92 + 1.25 * (16 + 8 + 32)) + 65536, used / (n * S)
        img = np.zeros((16, 16, 3), np.float32)
        cam = scenegen.frame_camera(v[..., :3].min((0, 1)), v[..., :3].max((0, 1)), 16, 16, perspective=True, fill=0.8)
        hr.hr_render(ctx, a, hr.render_desc(cam.pack(), scenegen.point_lights(1, np.zeros(3), seed=1), 1, 1, 1), img)
        assert img.max() > 0
    finally:
        hr.hr_destroy(ctx)
