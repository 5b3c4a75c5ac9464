"""The node boxes' grid is taken from the hair as it is, not as it was: node visits
of a counting frame equal those of an asset that never was elsewhere."""
import numpy as np
import pytest

import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu
RES = 48


def _asset(ctx, v):
    n = v.shape[0]
    return hr.hr_asset_create(ctx, v, scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2)),
                              np.zeros((n, 2), np.float32))


def _visits(ctx, a, v, lod=None):
    hr.hr_build_bvh(ctx, a, lod)
    cam = scenegen.frame_camera(v[..., :3].min((0, 1)), v[..., :3].max((0, 1)), RES, RES, perspective=True, fill=0.7)
    d = hr.render_desc(cam.pack(), scenegen.point_lights(1, np.zeros(3), seed=1), 4, 3, 1, 0, hr.HR_FLAG_COUNT)
    img = np.zeros((RES, RES, 3), np.float32)
    st = hr.hr_render(ctx, a, d, img, stats=True)
    assert img.max() > 0
    return st.node_visits, st.prim_tests, img


@pytest.mark.parametrize("n,S", [(300, 9), (24, 2100)])  # skinned in one pass; strands too long for it
def test_skinned_away_and_back(ctx, n, S):
    v = scenegen.make_strands(n, S, seed=3, jitter=0.002, hang=0.08, radius=4e-3)
    out = []
    for away in (False, True):
        a = _asset(ctx, v)
        hr.hr_build_guided_clusters(ctx, a, 5, 2)
        guides = np.zeros(5, np.int32)
        hr.hr_guides_export(ctx, a, guides)
        pose = np.ascontiguousarray(v[np.maximum(guides, 0)])
        if away:
            far = pose.copy()
            far[..., :3] += np.float32(20.0)
            hr.hr_asset_skin(ctx, a, far)
        hr.hr_asset_skin(ctx, a, pose)
        out.append(_visits(ctx, a, v))
        hr.hr_asset_destroy(ctx, a)
    assert out[0][:2] == out[1][:2] and np.array_equal(out[0][2], out[1][2])


@pytest.mark.parametrize("clusters", [300, 200])  # one strand or two a cluster: no thick hairs
def test_another_hierarchy_after_moving(ctx, clusters):
    v = scenegen.make_strands(300, 9, seed=3, jitter=0.002, hang=0.08, radius=4e-3)
    far = v.copy()
    far[..., :3] += np.float32(20.0)
    out = []
    for moved in (False, True):
        a = _asset(ctx, far if moved else v)
        if moved:
            hr.hr_build_clusters(ctx, a, 20)
            hr.hr_asset_update(ctx, a, v)
        hr.hr_build_clusters(ctx, a, clusters)
        assert hr.hr_hierarchy_info(ctx, a)[2] == 0
        out.append(_visits(ctx, a, v))
        hr.hr_asset_destroy(ctx, a)
    assert out[0][:2] == out[1][:2] and np.array_equal(out[0][2], out[1][2])


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_10565_gb300.build import build
    build()
    c = hr.hr_create(0)
    yield c
    hr.hr_destroy(c)
