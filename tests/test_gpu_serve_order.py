"""A request submitted right after API calls that return before their work is done
(device outputs, an update from device memory) is admitted after that work: it
renders the new positions, and its build shares no scratch with a frame still
under way."""
import numpy as np
import pytest
import torch

import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("clusters", [0, 300])
def test_requests_wait_for_the_calls_before_them(clusters):
    from paper_2405_10565_gb300.build import build
    build()
    n, S, W, H = 20000, 32, 160, 96
    v = scenegen.make_strands(n, S, seed=1, radius=2e-3)
    moved = v.copy()
    moved[..., 0] += np.linspace(0.0, 0.2, S + 1, dtype=np.float32)
    mat = scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2))
    cam = scenegen.frame_camera(v[..., :3].min((0, 1)), v[..., :3].max((0, 1)), W, H, perspective=True, fill=0.8).pack()
    lights = scenegen.point_lights(2, np.zeros(3), seed=1)
    d = hr.render_desc(cam, lights, 2, 2, 1)
    big = hr.render_desc(scenegen.frame_camera(v[..., :3].min((0, 1)), v[..., :3].max((0, 1)), 1280, 720,
                                               perspective=True, fill=0.8).pack(), lights, 8, 4, 1)
    ctx = hr.hr_create(0)
    try:
        poses = [torch.from_numpy(p).cuda() for p in (v, moved)]
        a, other = (hr.hr_asset_create(ctx, v, mat, np.zeros((n, 2), np.float32)) for _ in range(2))
        out = torch.zeros(720, 1280, 3, device="cuda")
        want = []
        for p in poses:
            hr.hr_asset_update(ctx, a, p)
            if clusters:
                hr.hr_build_clusters(ctx, a, clusters)
                hr.hr_select_lod(ctx, a, cam, 2.0, 0, 0, None)
            hr.hr_build_bvh(ctx, a, None)
            want.append(np.zeros((H, W, 3), np.float32))
            hr.hr_render(ctx, a, d, want[-1])
        assert np.linalg.norm(want[1] - want[0]) > 0.1 * np.linalg.norm(want[0])
        torch.cuda.synchronize()
        hr.hr_serve_start(ctx, 2, 1 << 22)
        try:
            for i in range(6):
                if clusters:  # the hierarchy of the pose, ready; then its strands once more
                    hr.hr_asset_update(ctx, a, poses[i % 2])
                    hr.hr_build_clusters(ctx, a, clusters)
                for _ in range(3):
                    hr.hr_render_frame(ctx, other, 0, 2.0, 0, big, out)
                hr.hr_asset_update(ctx, a, poses[i % 2])
                img = np.full((H, W, 3), 7.0, np.float32)
                st, res = hr.hr_poll(ctx, hr.hr_submit(ctx, a, d, img, 2.0, 0), 60000)
                assert st == hr.HR_OK and res.status == hr.HR_OK
                # the bound of the served mixes
                assert np.linalg.norm(img - want[i % 2]) <= 1e-5 * np.linalg.norm(want[i % 2]), i
        finally:
            hr.hr_serve_stop(ctx)
    finally:
        hr.hr_destroy(ctx)
