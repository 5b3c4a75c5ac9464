"""Scenes with odd vertices.  One that is not a number or infinite: the
segments that touch it are never hit, and every other segment is, as the oracle
has it without them.  One far away, or parts of very different scale, which the
node boxes' grid does not resolve: as the oracle has the scene, and at the cost
of the same scene without it."""
import numpy as np
import pytest

import oracle
import paper_2405_10565_gb300 as hr
import scenegen
from gpu_util import HIT_AGREE_MIN, KBUF_AGREE_MIN, RMSE_FP32, compare, gpu_samples

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_10565_gb300.build import build
    build()
    c = hr.hr_create(0)
    yield c
    hr.hr_destroy(c)


def _scene(n, S, seed=1):
    v = scenegen.make_strands(n, S, seed=seed, jitter=0.01, radius=4e-3)
    return scenegen.Scene(v, scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2)),
                          np.stack([np.full(n, 0.7), np.linspace(0, 6, n)], -1).astype(np.float32))


def _check(ctx, sc, odd, bad, update, fill=0.8, res=40, k=3, spp=2):
    """Render `sc` with its vertices replaced by `odd`; `bad` marks the
    vertices whose segments the oracle leaves out."""
    n, S = sc.n_strands, sc.n_segments
    cam = scenegen.frame_camera(*sc.aabb(), res, res, perspective=True, fill=fill)
    lights = scenegen.point_lights(2, 0.5 * sum(sc.aabb()), seed=2)
    clean = np.where(bad[..., None], sc.verts, odd)
    rows, ids = oracle.strand_prim_rows(clean, sc.shape, np.arange(n))
    keep = ~(bad[:, :-1] | bad[:, 1:]).reshape(-1)
    prep = oracle.Prepared(np.ascontiguousarray(rows[keep]), np.ascontiguousarray(ids[keep].astype(np.int64)),
                           sc.mat.astype(np.float64), None, None, None)
    a = hr.hr_asset_create(ctx, sc.verts if update else odd, sc.mat, sc.shape)
    try:
        if update:
            hr.hr_asset_update(ctx, a, odd)
        hr.hr_build_bvh(ctx, a, None)
        d = hr.render_desc(cam.pack(), lights, spp, k, 5)
        sids = np.arange(res * res * spp)
        rg, hg = gpu_samples(ctx, a, d, sids)
        ro, ho = oracle.render_samples(prep, cam.pack(), lights, sids, spp, k, 5)
        near, full, rel, _ = compare(rg, hg, ro, ho)
        assert (ho[:, 0] >= 0).any()
        assert near >= HIT_AGREE_MIN and full >= KBUF_AGREE_MIN and rel <= RMSE_FP32, (near, full, rel)
        img = np.zeros((res, res, 3), np.float32)
        hr.hr_render(ctx, a, d, img)
        mean = rg.reshape(-1, spp, 3).astype(np.float64).mean(1).reshape(img.shape)
        assert np.allclose(img, mean, rtol=1e-4, atol=1e-6 * max(1.0, float(mean.max())))
    finally:
        hr.hr_asset_destroy(ctx, a)


@pytest.mark.parametrize("update", [False, True])
@pytest.mark.parametrize("n,S", [(40, 8), (300, 8)])  # a BVH of one block; of several
@pytest.mark.parametrize("vertex,axes", [(0, (0, 1, 2)), (0, (1,)), (4, (0, 1, 2)), (8, (2,))])
def test_a_vertex_that_is_not_a_number(ctx, n, S, vertex, axes, update):
    sc = _scene(n, S)
    odd, bad = np.array(sc.verts), np.zeros((n, S + 1), bool)
    for s in (n // 3, n - 1):
        odd[s, vertex, list(axes)] = np.nan
        bad[s, vertex] = True
    _check(ctx, sc, odd, bad, update)


@pytest.mark.parametrize("n,S", [(40, 8), (300, 8)])
@pytest.mark.parametrize("vertex,value", [(0, np.inf), (8, -np.inf), (4, np.inf)])
def test_an_infinite_vertex(ctx, n, S, vertex, value):
    sc = _scene(n, S)
    odd, bad = np.array(sc.verts), np.zeros((n, S + 1), bool)
    odd[n // 2, vertex, 1] = value
    bad[n // 2, vertex] = True
    _check(ctx, sc, odd, bad, False)


def _far(sc, distance, vertex=-1):
    odd = np.array(sc.verts)
    odd[odd.shape[0] // 2, vertex, :3] += np.asarray([1.0, 0.3, -1.0], np.float32) * distance
    return odd


@pytest.mark.parametrize("n,S", [(40, 8), (300, 8)])
@pytest.mark.parametrize("distance", [30.0, 1e3, 1e5, 1e9])  # the grid resolves the first alone
def test_a_vertex_far_away(ctx, n, S, distance):
    sc = _scene(n, S)
    _check(ctx, sc, _far(sc, distance), np.zeros((n, S + 1), bool), False)


@pytest.mark.parametrize("parts,ratio", [(2, 1e4), (3, 100.0)])
def test_parts_of_very_different_scale_or_far_apart(ctx, parts, ratio):
    """Two heads 10,000 heads apart; three of scales 1, 1 / 100 and 1 / 10,000
    side by side.  The camera sees the first."""
    sc = _scene(300, 8)
    n = sc.n_strands
    odd = np.array(sc.verts)
    for p in range(1, parts):
        part = slice(p * n // parts, (p + 1) * n // parts)
        if parts == 2:
            odd[part, :, :3] += np.asarray([0.0, 0.0, ratio], np.float32)
        else:
            odd[part, :, :3] = odd[part, :, :3] * ratio ** -p + np.asarray([1.5 * p, 0.0, 0.0], np.float32)
            odd[part, :, 3] *= ratio ** -p
    _check(ctx, sc, odd, np.zeros((n, 9), bool), False)


@pytest.mark.parametrize("settled", ["built", "refit"])
@pytest.mark.parametrize("distance", [1e3, 1e5])
def test_a_far_vertex_costs_little(ctx, distance, settled):
    """Node visits of a counting frame of 3,000 strands (clustered, so that the
    list of leaves is in order): without the far vertex 1, with it below 2."""
    w = scenegen.clustered(n=3000, S=16, res=96, spp=2, lod_setting="strands", n_clusters=60)
    sc = w.scene
    img = np.zeros((96, 96, 3), np.float32)
    visits = []
    for verts in (sc.verts, _far(sc, distance)):
        a = hr.hr_asset_create(ctx, sc.verts, sc.mat, sc.shape)
        hr.hr_build_clusters(ctx, a, w.n_clusters)
        C, L, _ = hr.hr_hierarchy_info(ctx, a)
        lod = scenegen.lod_preset("strands", C, L)
        if settled == "refit":
            hr.hr_build_bvh(ctx, a, lod)
        hr.hr_asset_update(ctx, a, verts)
        flags = hr.HR_FLAG_COUNT
        if settled == "built":
            hr.hr_build_bvh(ctx, a, lod)
            st = hr.hr_render(ctx, a, hr.render_desc(w.camera.pack(), w.lights, 2, 4, 7, 0, flags), img, stats=True)
        else:
            flags |= hr.HR_FLAG_REFIT | hr.HR_FLAG_KEEP_HIERARCHY
            d = hr.render_desc(w.camera.pack(), w.lights, 2, 4, 7, 0, flags)
            st = hr.hr_render_frame(ctx, a, 0, 0.0, 0, d, img, stats=True)
        visits.append(st.node_visits / max(1, st.traced_samples))
        hr.hr_asset_destroy(ctx, a)
    print(settled, distance, visits)
    assert 0 < visits[1] < 2 * visits[0]
