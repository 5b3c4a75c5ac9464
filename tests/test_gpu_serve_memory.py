"""A request is admitted where the memory it needs is only held by what frames can
do without (room for rays put aside, light paths)."""
import numpy as np
import pytest

import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, hr.HR_FLAG_SHADOWS])
def test_serving_reclaims_what_frames_can_do_without(flags):
    from paper_2405_10565_gb300.build import build
    build()
    n, S, W, H = 2500, 16, 640, 400
    v = scenegen.make_strands(n, S, seed=1, radius=4e-3)
    mat = scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2))
    cam = scenegen.frame_camera(v[..., :3].min((0, 1)), v[..., :3].max((0, 1)), W, H, perspective=True, fill=0.8)
    lights = scenegen.point_lights(2, np.zeros(3), seed=1)
    frame = hr.render_desc(cam.pack(), lights, 8, 4, 1, 0, flags)
    served = hr.render_desc(cam.pack(), lights, 2, 4, 1)

    def set_up(budget):
        ctx = hr.hr_create(0, budget)
        a = hr.hr_asset_create(ctx, v, mat, np.zeros((n, 2), np.float32))
        hr.hr_build_bvh(ctx, a, None)
        before = hr.hr_bytes_in_use(ctx)
        img = np.zeros((H, W, 3), np.float32)
        hr.hr_render(ctx, a, frame, img)
        return ctx, a, img, hr.hr_bytes_in_use(ctx) - before, hr.hr_bytes_in_use(ctx)

    ctx, _, _, taken, used = set_up(0)
    hr.hr_destroy(ctx)
    assert taken > 16 << 20  # far more than the request needs
    ctx, a, img, _, again = set_up(used + (1 << 20))
    try:
        assert again == used and img.max() > 0
        want = np.zeros((H, W, 3), np.float32)
        hr.hr_serve_start(ctx, 1, 1 << 22)
        try:
            out = np.full((H, W, 3), 7.0, np.float32)
            st, res = hr.hr_poll(ctx, hr.hr_submit(ctx, a, served, out, 2.0, 0), 60000)
            assert st == hr.HR_OK and res.status == hr.HR_OK
        finally:
            hr.hr_serve_stop(ctx)
        hr.hr_render(ctx, a, served, want)
        assert np.linalg.norm(out - want) <= 1e-5 * np.linalg.norm(want)
    finally:
        hr.hr_destroy(ctx)
