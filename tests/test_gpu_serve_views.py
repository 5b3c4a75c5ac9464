"""Served images against hr_render where the scene's projected rectangle can go
wrong: scene across the image's edge, out of view, behind the eye and around
it, perspective and orthographic, a first request of a BVH and later ones."""
import dataclasses

import numpy as np
import pytest

import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("perspective", [True, False])
def test_views_at_the_edges_of_the_scene_rectangle(perspective):
    from paper_2405_10565_gb300.build import build
    build()
    W, H = 61, 43
    w = scenegen.full_head(n=800, S=8, width=W, height=H, spp=2, n_lights=2, n_clusters=32, seed=4)
    lo, hi = w.scene.aabb()
    base = scenegen.frame_camera(lo, hi, W, H, perspective=perspective, fill=0.6)
    size = float(np.max(hi - lo))
    mid = 0.5 * (np.asarray(lo) + np.asarray(hi))
    eyes = [base.eye,
            base.eye + 0.5 * size * base.right,               # across an edge
            base.eye + 0.8 * size * (base.right + base.up),   # across a corner
            base.eye + 50.0 * size * base.right,              # out of view
            mid,                                              # inside
            base.eye + 100.0 * size * base.fwd]               # behind the eye
    cams = [dataclasses.replace(base, eye=e) for e in eyes]
    ctx = hr.hr_create(0)
    try:
        a = hr.hr_asset_create(ctx, w.scene.verts, w.scene.mat, w.scene.shape)
        hr.hr_build_clusters(ctx, a, w.n_clusters)
        C, _, _ = hr.hr_hierarchy_info(ctx, a)
        descs = [hr.render_desc(c.pack(), w.lights, 2, 3, 11, 0) for c in cams]
        ref = []
        for c, d in zip(cams, descs):
            lod = np.zeros(C, np.uint8)
            hr.hr_select_lod(ctx, a, c.pack(), 2.0, 0, 0, lod)
            hr.hr_build_bvh(ctx, a, lod)
            ref.append(np.zeros((H, W, 3), np.float32))
            hr.hr_render(ctx, a, d, ref[-1])
        assert ref[0].max() > 0 and ref[1].max() > 0 and ref[4].max() > 0 and ref[3].max() == 0
        hr.hr_serve_start(ctx, 3, 1 << 20)
        try:
            for _ in range(2):  # the second pass finds the BVHs resident
                out = [np.full((H, W, 3), 7.0, np.float32) for _ in cams]
                tickets = [hr.hr_submit(ctx, a, d, o, 2.0, 0) for d, o in zip(descs, out)]
                for t in tickets:
                    st, res = hr.hr_poll(ctx, t, 60000)
                    assert st == hr.HR_OK and res.status == hr.HR_OK
                # the same operations; two kernels, which the compiler may contract
                # differently: the bound of the served mixes
                for o, r in zip(out, ref):
                    assert np.linalg.norm(o - r) <= 1e-5 * np.linalg.norm(r)
        finally:
            hr.hr_serve_stop(ctx)
    finally:
        hr.hr_destroy(ctx)
